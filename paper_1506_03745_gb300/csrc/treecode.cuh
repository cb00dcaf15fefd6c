// Treecode kernels of the boundary-element matvec (Section 3.2 of the paper),
// templated on the arithmetic type and on the Taylor order P.
//
// Combined potential.  Every row of Eq. 6 / Eq. 7 needs, per target x and per
// kernel G (Laplace 1/r or Yukawa e^{-kappa r}/r, without the 1/4pi), the
// combination U = S_V - S_K of single- and double-layer sums:
//   U(x) = sum_s [ q_s G(x - y_s) - p_s . grad_y G(x - y_s) ],
// with, per quadrature point s of panel j (weight w_s = w_m A_j):
//   q_s = w_s psi_j  (single-layer density),  p_s = w_s phi_j n_j (double layer).
// Near: direct sum.  Far: G(R - d) = sum_k G_k(R) (-d)^k with R = x - c,
// d = y - c, G_k = d^k G / k! (derivatives in R), so
//   U = sum_k G_k(R) M_k,  M_k = sum_s (q_s + p_s . grad_u) u_s^k,  u_s = c - y_s.
// Recurrences for G_k (derived from rho^2 dG/dR_i = -R_i G - kappa R_i H and
// dH/dR_i = -kappa R_i G with H = e^{-kappa rho}), n = |k| >= 1:
//   S1 = sum_a R_a G_{k-e_a},  S2 = sum_a G_{k-2e_a}   (and T1, T2 with H)
//   H_k = -(kappa/n) (S1 + S2)
//   G_k = -[(2n-1) S1 + (n-1) S2 + kappa (T1 + T2)] / (n rho^2)
// Laplace is the same with kappa = 0 (H_0 = 1, H_k = 0).
// Moment shift (upward pass): M_k(c') = sum_{j<=k} C(k,j) (c'-c)^{k-j} M_j(c).
#pragma once
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "ds.cuh"
#include "pgb_internal.cuh"

namespace pgb {

struct __align__(16) ds4 {
    ds x, y, z, w;
};

template <typename T>
struct V4;
template <>
struct V4<float> {
    using t = float4;
};
template <>
struct V4<double> {
    using t = dbl4;
};
template <>
struct V4<ds> {
    using t = ds4;
};

// Storage type of the kernels' inputs per arithmetic type: the
// double-single kernels read the FP64 product's data (source terms, target
// offsets, moments) and convert as they stage it.
template <typename C>
struct Store {
    using S = C;
};
template <>
struct Store<ds> {
    using S = double;
};
template <typename C>
__device__ __forceinline__ C to_c(typename Store<C>::S v) {
    return v;
}
template <>
__device__ __forceinline__ ds to_c<ds>(double v) {
    return ds_from_double(v);
}
template <typename C>
__device__ __forceinline__ typename V4<C>::t cvt4(const typename V4<typename Store<C>::S>::t& v) {
    return v;
}
template <>
__device__ __forceinline__ ds4 cvt4<ds>(const dbl4& v) {
    return ds4{ds_from_double(v.x), ds_from_double(v.y), ds_from_double(v.z), ds_from_double(v.w)};
}
__device__ __forceinline__ double to_dbl(float v) { return (double)v; }
__device__ __forceinline__ double to_dbl(double v) { return v; }
__device__ __forceinline__ double to_dbl(ds v) { return ds_to_double(v); }
// a double in the arithmetic type
template <typename real>
__device__ __forceinline__ real from_dbl(double v) {
    return (real)v;
}
template <>
__device__ __forceinline__ ds from_dbl<ds>(double v) {
    return ds_from_double(v);
}

// a double literal in the arithmetic type (split at compile time for ds)
template <typename C>
__device__ __forceinline__ C lit(double d) {
    return (C)d;
}
template <>
__device__ __forceinline__ ds lit<ds>(double d) {
    return ds_const(d);
}

__device__ __forceinline__ float rsqrt_(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_(double x) { return rsqrt_halley(x); }
__device__ __forceinline__ float exp_(float x) { return __expf(x); }
__device__ __forceinline__ double exp_(double x) { return exp(x); }
// 2^x (the P2P loop folds log2(e) into its constant) and 1/sqrt(x) of the
// P2P loop.  FP32: the SFU's approximate forms (relative error about 2^-22),
// one instruction each.  FP64: exp2_table and rsqrt_halley (relative errors
// below 1e-14 and of FP64 rounding), about a quarter of the FP64 operations of
// the library's correctly rounded forms on a part whose FP64 rate is 1/64 of
// its FP32 rate.
__device__ __forceinline__ float exp2_(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ double exp2_(double x) { return exp2_table(x); }
__device__ __forceinline__ float rsqrt_fast(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ double rsqrt_fast(double x) { return rsqrt_halley(x); }
__device__ __forceinline__ ds rsqrt_(ds x) { return ds_rsqrt(x); }
__device__ __forceinline__ ds rsqrt_fast(ds x) { return ds_rsqrt(x); }
__device__ __forceinline__ ds exp_(ds x) { return ds_exp(x); }
__device__ __forceinline__ ds exp2_(ds x) { return ds_exp2(x); }

// Neumaier-compensated accumulation s + c += v.
template <typename T>
__device__ __forceinline__ void kadd(T& s, T& c, T v) {
    T t = s + v;
    c += (fabs(s) >= fabs(v)) ? ((s - t) + v) : ((v - t) + s);
    s = t;
}
// double-single sums carry their own error term (c stays 0)
__device__ __forceinline__ void kadd(ds& s, ds&, ds v) { s = s + v; }

// c + a b: as written for FP32 / FP64 (the compiler contracts it), one fused
// double-single operation for ds
template <typename T>
__device__ __forceinline__ T madd(T a, T b, T c) {
    return c + a * b;
}
__device__ __forceinline__ ds madd(ds a, ds b, ds c) { return ds_fma(a, b, c); }
template <typename T>
constexpr bool is_ds = false;
template <>
constexpr bool is_ds<ds> = true;

// Arithmetic of the P2P and M2P sums.
__device__ __forceinline__ float mul_(float a, float b) { return a * b; }
__device__ __forceinline__ double mul_(double a, double b) { return a * b; }
__device__ __forceinline__ float add_(float a, float b) { return a + b; }
__device__ __forceinline__ double add_(double a, double b) { return a + b; }
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
// Two FP32 values in one 64-bit register pair: Blackwell's packed FP32
// arithmetic does both with one instruction.  The FMA pipe takes as long as
// for two scalar ones (measured: 113-118 lane FMAs per clock and SM either
// way); what halves is the issue slots.
struct __align__(8) f2 {
    float a, b;
};
__device__ __forceinline__ unsigned long long f2_bits(f2 x) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x.a), "f"(x.b));
    return r;
}
__device__ __forceinline__ f2 f2_from(unsigned long long v) {
    f2 x;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x.a), "=f"(x.b) : "l"(v));
    return x;
}
__device__ __forceinline__ f2 mul_(f2 x, f2 y) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(x)), "l"(f2_bits(y)));
    return f2_from(r);
}
__device__ __forceinline__ f2 add_(f2 x, f2 y) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(x)), "l"(f2_bits(y)));
    return f2_from(r);
}
__device__ __forceinline__ f2 fma_(f2 x, f2 y, f2 z) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_bits(x)), "l"(f2_bits(y)), "l"(f2_bits(z)));
    return f2_from(r);
}
__device__ __forceinline__ f2 operator-(f2 x) { return f2{-x.a, -x.b}; }
__device__ __forceinline__ f2 rsqrt_(f2 x) { return f2{rsqrt_(x.a), rsqrt_(x.b)}; }
__device__ __forceinline__ f2 exp_(f2 x) { return f2{exp_(x.a), exp_(x.b)}; }
// a constant in the arithmetic type
template <typename V>
__device__ __forceinline__ V cst(double d) {
    return (V)d;
}
template <>
__device__ __forceinline__ f2 cst<f2>(double d) {
    return f2{(float)d, (float)d};
}

// Multi-indices of total degree <= P: graded, and within a degree kx
// descending then ky descending.
template <int P>
struct MI {
    static constexpr int T = (P + 1) * (P + 2) * (P + 3) / 6;
    int k[T][3];
    int lvl[T];
    int m1[T][3];
    int m2[T][3];
    constexpr MI() : k(), lvl(), m1(), m2() {
        int t = 0;
        for (int n = 0; n <= P; ++n)
            for (int x = n; x >= 0; --x)
                for (int y = n - x; y >= 0; --y) {
                    k[t][0] = x;
                    k[t][1] = y;
                    k[t][2] = n - x - y;
                    lvl[t] = n;
                    ++t;
                }
        for (int i = 0; i < T; ++i)
            for (int a = 0; a < 3; ++a) {
                m1[i][a] = -1;
                m2[i][a] = -1;
                for (int j = 0; j < T; ++j) {
                    bool e1 = true, e2 = true;
                    for (int b = 0; b < 3; ++b) {
                        int d = (a == b) ? 1 : 0;
                        if (k[j][b] != k[i][b] - d) e1 = false;
                        if (k[j][b] != k[i][b] - 2 * d) e2 = false;
                    }
                    if (e1) m1[i][a] = j;
                    if (e2) m2[i][a] = j;
                }
            }
    }
    constexpr int index(int x, int y, int z) const {
        for (int i = 0; i < T; ++i)
            if (k[i][0] == x && k[i][1] == y && k[i][2] == z) return i;
        return -1;
    }
};

// Runtime decode of the multi-index order of MI<P>: index t -> (kx, ky, kz).
__device__ __forceinline__ void decode_mi(int t, int& x, int& y, int& z) {
    int n = 0, cnt = 1;
    while (t >= cnt) {
        t -= cnt;
        ++n;
        cnt = (n + 1) * (n + 2) / 2;
    }
    int xx = n, m = 1;
    while (t >= m) {
        t -= m;
        --xx;
        ++m;
    }
    x = xx;
    y = (n - xx) - t;
    z = n - x - y;
}

// the run-time body mask of a product (all bodies without one)
__device__ __forceinline__ unsigned long long body_mask(const unsigned long long* m) { return m ? *m : ~0ull; }

// stage code of the panel moments' launch (the others: PGB_STAGE_*)
#define STAGE_PANEL_MOMENTS (-1)

struct EvalArgs {
    int64_t n_pan;
    const int32_t *gstart, *gend, *gbody;
    const double* gcenter;
    const int64_t *near_off, *far_off;
    const int32_t *near_l, *far_l;
    const int32_t *nstart, *nend, *nbody;
    const double* ncenter;
    int K;
    double kappa;
    int lap_body[PGB_MAX_BODIES];  // 1 when the body is dielectric
    int src_active[PGB_MAX_BODIES];  // 0: the body's densities are all zero (skip)
    int all_active;                // every body active (the plain product): no per-node test
    unsigned long long tgt_mask;   // bit b: the rows of body b are used (other groups' items are skipped)
    int64_t g_lo, g_hi;            // only the groups g_lo <= g < g_hi (a rank's rows of a sharded product)
    // device copy of a further body mask, read at run time (a replayed
    // lockstep iteration: bit b clear = body b's rows and sources left out);
    // nullptr: none.  With it all_active is 0.
    const unsigned long long* bmask = nullptr;
    const float4* far4;            // per far entry: node centre - group centre, node id bits
    const int64_t* col_off;        // per group: its P2P columns [col_off[g], col_off[g+1])
    const float4* col;             // per column: panel centroid - group centre (FP32), panel (int bits); nullptr:
    const int32_t* ent_col;        // not kept, found by each near entry's first column in its group
    const double* cen;             // panel centroids
    const int32_t* pnode;          // leaf node of a panel (FP64 and double-single offsets)
    const int32_t* pbody;          // body of a panel
    const void* pg;                // panel geometry (PanelGeo) in the kernel's arithmetic (FP64 for double-single)
    const void* pd;                // panel densities x area, same arithmetic: {psiL, psiY, phi, unused}
    const dbl4* pts;               // double-single: the far rule's points relative to their leaf's centre
    const void *near_mat = nullptr, *near_group = nullptr;  // stored near field (solves), nullptr: formed
    FarRule rule;
    unsigned long long src_mask;   // bit b: src_active[b]
    // work items (a group's columns in even runs, its far entries in runs of m2p_item)
    int64_t n_pitems, n_fitems;
    const int64_t *pitem_off, *fitem_off;  // per group
    const int32_t *pitem_group, *fitem_group;
    double *Up, *Uf;               // per item: 32 Laplace then 32 Yukawa partial sums (one per lane)
    // persistent launch: a grid smaller than the item count whose blocks take
    // items from these counters (zero before the launch); nullptr: one item per block
    unsigned long long *p2p_work, *m2p_work;
    int persist_blocks;            // grid of a persistent launch
};

// Column i of group g, whose columns start at c0 (EvalArgs::col).  Without the
// table the near entry that holds it is searched for, and the offset formed as
// the table's is.
__device__ __forceinline__ float4 column(const EvalArgs& a, int64_t g, int64_t c0, int64_t i) {
    if (a.col) return a.col[c0 + i];
    int64_t lo = a.near_off[g], hi = a.near_off[g + 1];
    while (hi - lo > 1) {
        const int64_t m = (lo + hi) >> 1;
        if (a.ent_col[m] <= i) lo = m;
        else hi = m;
    }
    const int64_t j = a.nstart[a.near_l[lo]] + (i - a.ent_col[lo]);
    return make_float4((float)(a.cen[3 * j] - a.gcenter[3 * g]), (float)(a.cen[3 * j + 1] - a.gcenter[3 * g + 1]),
                       (float)(a.cen[3 * j + 2] - a.gcenter[3 * g + 2]), __int_as_float((int)j));
}

// Item loop of a block: one item per block, or (persistent launch) items
// taken from a counter until none is left.  The barrier also keeps a block
// from reusing its shared memory while a warp still reads the last item.
__device__ __forceinline__ int64_t next_item(unsigned long long* work, int64_t cur, int64_t* slot) {
    if (!work) return cur < 0 ? (int64_t)blockIdx.x : INT64_MAX;
    __syncthreads();
    if (threadIdx.x == 0) *slot = (int64_t)atomicAdd(work, 1ull);
    __syncthreads();
    return *slot;
}

// 16-byte vector of the arithmetic type (4 floats, 2 doubles, 2 double-singles),
// for loads of consecutive coefficients from shared memory.
template <typename real>
struct alignas(16) Vec16 {
    static constexpr int N = 16 / sizeof(real);
    real v[N];
};

// Compile-time loop: f(std::integral_constant<int, I>) for I = B .. E-1, so
// that array indices formed from I are constants whatever the trip count
// (a plain unrolled loop nest is left partly rolled by the compiler at the
// higher orders, which moves the per-degree sums to local memory).
template <int B, int E, class F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (B < E) {
        f(std::integral_constant<int, B>{});
        static_for<B + 1, E>(f);
    }
}
// Position of the coefficient (l, m, s) among a node's: m = 0 first, then per
// m the (Re, Im) pairs of l = m..P.
__host__ __device__ constexpr int far_pos(int P, int l, int m, int s) {
    return m == 0 ? l : (P + 1) + 2 * ((m - 1) * (P + 1) - (m - 1) * m / 2) + 2 * (l - m) + s;
}
// c_{l,m} of the q recurrence
__host__ __device__ constexpr double far_c(int l, int m) { return (double)(l * l - m * m) / (4.0 * l * l - 1.0); }

// Far field of one node at R = target - node centre from its harmonic
// coefficients (farfield.cu), n = R / r, x = kappa r:
//   U_Y = (e^{-x} / r) sum_l h_l sum_m q_{l,m}(n_z) (a Re + b Im)(n_x + i n_y)^m,
//   U_L = (1 / r) sum_l r^{-l} sum_m ...,
// h_l = g_l(x) r^{-l}: h_0 = 1, h_1 = -(1 + x) / r, h_l = kappa^2 h_{l-2} -
// (2l - 1) h_{l-1} / r.  Unrolled at compile time, so that the radial factors
// stay in registers.  V: the arithmetic (f2: two targets); C: the stored
// constants' type, the recurrence constants -c_{l,m} at ctab[l (P + 1) + m] for
// f2 (packed instructions take no immediates), immediate otherwise.
template <typename V, int P, bool LAP>
__device__ __forceinline__ void far_eval(V Rx, V Ry, V Rz, V kappa, const V* __restrict__ cL,
                                         const V* __restrict__ cY, const V* __restrict__ ctab, V& uL, V& uY) {
    using W = Vec16<V>;
    constexpr int VN = W::N;
    constexpr bool PACKED = std::is_same<V, f2>::value;
    V hY[P + 1], hL[P + 1];
    const V r2 = fma_(Rz, Rz, fma_(Ry, Ry, mul_(Rx, Rx)));
    const V ri = rsqrt_(r2);
    const V nx = mul_(Rx, ri), ny = mul_(Ry, ri), nz = mul_(Rz, ri);
    const V ex = mul_(exp_(mul_(-kappa, mul_(r2, ri))), ri);
    const V k2 = mul_(kappa, kappa);
    hY[0] = hL[0] = cst<V>(1);
    if constexpr (P >= 1) {
        hY[1] = -add_(ri, kappa);  // -(1 + x) / r
        hL[1] = ri;
    }
    V lr = ri;  // (2l - 1) / r
    const V twice = add_(ri, ri);
    static_for<2, P + 1>([&](auto Lc) {
        constexpr int l = decltype(Lc)::value;
        lr = add_(lr, twice);
        hY[l] = fma_(-lr, hY[l - 1], mul_(k2, hY[l - 2]));
        if constexpr (LAP) hL[l] = mul_(hL[l - 1], ri);
    });
    V X = cst<V>(1), Y = cst<V>(0);
    uL = uY = cst<V>(0);
    W qy, ql;
    static_for<0, P + 1>([&](auto M) {
        constexpr int m = decltype(M)::value;
        V q0 = cst<V>(1), q1 = cst<V>(0);  // q_{l,m}, q_{l-1,m}
        V aY, bY, aL, bL;                  // the sums over l
        static_for<m, P + 1>([&](auto Lc) {
            constexpr int l = decltype(Lc)::value;
            if constexpr (l > m) {
                V q;
                if constexpr (l == m + 1) q = nz;
                else if constexpr (PACKED) q = fma_(nz, q0, mul_(ctab[(l - 1) * (P + 1) + m], q1));
                else q = fma_(nz, q0, mul_(cst<V>(-far_c(l - 1, m)), q1));
                q1 = q0;
                q0 = q;
            }
            V w, v;
            if constexpr (l > m) {
                w = mul_(hY[l], q0);
                if constexpr (LAP) v = mul_(hL[l], q0);
            } else {
                w = hY[l];
                if constexpr (LAP) v = hL[l];
            }
            static_for<0, (m == 0 ? 1 : 2)>([&](auto Sc) {
                constexpr int s = decltype(Sc)::value;
                constexpr int i = far_pos(P, l, m, s);
                if constexpr (i % VN == 0) {
                    qy = *reinterpret_cast<const W*>(cY + i);
                    if constexpr (LAP) ql = *reinterpret_cast<const W*>(cL + i);
                }
                V& sy = s == 0 ? aY : bY;
                if constexpr (l == m) sy = mul_(w, qy.v[i % VN]);
                else sy = fma_(w, qy.v[i % VN], sy);
                if constexpr (LAP) {
                    V& sl = s == 0 ? aL : bL;
                    if constexpr (l == m) sl = mul_(v, ql.v[i % VN]);
                    else sl = fma_(v, ql.v[i % VN], sl);
                }
            });
        });
        if constexpr (m == 0) {
            uY = aY;
            if constexpr (LAP) uL = aL;
            X = nx;
            Y = ny;
        } else {
            uY = fma_(X, aY, fma_(Y, bY, uY));
            if constexpr (LAP) uL = fma_(X, aL, fma_(Y, bL, uL));
            if constexpr (m < P) {
                const V xn = fma_(nx, X, -mul_(ny, Y));
                Y = fma_(nx, Y, mul_(ny, X));
                X = xn;
            }
        }
    });
    uY = mul_(ex, uY);
    if constexpr (LAP) uL = mul_(ri, uL);
}

// c_{l,m} in double-single for the rolled form below
struct FarC {
    ds v[PGB_MAX_P + 1][PGB_MAX_P + 1];  // [m][l]
    __host__ __device__ constexpr FarC() : v() {
        for (int m = 0; m <= PGB_MAX_P; ++m)
            for (int l = 1; l <= PGB_MAX_P; ++l) v[m][l] = ds_const(far_c(l, m));
    }
};
__device__ __constant__ const FarC kFarC = FarC();

// The same in double-single, as loops: unrolled, a pair's 2500 operations
// overflow the instruction caches (the kernel waited for instructions more
// than for anything else).  rad: the thread's radial factors in shared memory,
// (h_l, r^{-l}) at rad[l * stride].
template <int P, bool LAP>
__device__ __forceinline__ void far_eval_ds(ds Rx, ds Ry, ds Rz, ds kappa, const ds* __restrict__ cL,
                                            const ds* __restrict__ cY, float4* rad, int stride, ds& uL, ds& uY) {
    const ds r2 = ds_norm(ds_fma_u(Rx, Rx, ds_fma_u(Ry, Ry, ds_mul_u(Rz, Rz))));
    const ds ri = ds_rsqrt(r2);
    const ds nx = Rx * ri, ny = Ry * ri, nz = Rz * ri;
    const ds ex = ds_mul_u(ds_exp(-(kappa * (r2 * ri))), ri);
    {
        const ds k2 = kappa * kappa;
        ds h0 = ds(1), h1 = -(ri + kappa), p = ds(1);
        rad[0] = make_float4(1.f, 0.f, 1.f, 0.f);
#pragma unroll 1
        for (int l = 1; l <= P; ++l) {
            if (l > 1) {
                // both terms carry the sign (-1)^l: no cancellation
                const ds h = ds_norm(ds_fma_u(k2, h0, ds_mul_u(mul_f(ri, -(float)(2 * l - 1)), h1)));
                h0 = h1;
                h1 = h;
            }
            p = p * ri;
            rad[l * stride] = make_float4(h1.hi, h1.lo, p.hi, p.lo);
        }
    }
    ds X = ds(1), Y = ds(0);
    ds sY = ds(0), sL = ds(0);
    int i = 0;
#pragma unroll 1
    for (int m = 0; m <= P; ++m) {
        ds q0 = ds(1), q1 = ds(0), aY = ds(0), bY = ds(0), aL = ds(0), bL = ds(0);
#pragma unroll 1
        for (int l = m; l <= P; ++l) {
            const float4 h = rad[l * stride];
            const ds w = ds_mul_u(ds(h.x, h.y), q0);
            aY = ds_fma_u(w, cY[i], aY);
            if (m) bY = ds_fma_u(w, cY[i + 1], bY);
            if (LAP) {
                const ds v = ds_mul_u(ds(h.z, h.w), q0);
                aL = ds_fma_u(v, cL[i], aL);
                if (m) bL = ds_fma_u(v, cL[i + 1], bL);
            }
            i += m ? 2 : 1;
            const ds q = nz * q0 - kFarC.v[m][l] * q1;  // c_{m,m} = 0
            q1 = q0;
            q0 = q;
        }
        sY = ds_fma_u(X, ds_norm(aY), ds_fma_u(Y, ds_norm(bY), sY));
        if (LAP) sL = ds_fma_u(X, ds_norm(aL), ds_fma_u(Y, ds_norm(bL), sL));
        const ds xn = nx * X - ny * Y;
        Y = nx * Y + ny * X;
        X = xn;
    }
    uY = ex * ds_norm(sY);
    uL = LAP ? ri * ds_norm(sL) : ds(0);
}

// e^{-kappa r} of the P2P sums as exp2_scaled(exp_scale(kappa), r).
__device__ __forceinline__ float exp_scale(float kappa) { return -kappa * 1.4426950408889634f; }
__device__ __forceinline__ double exp_scale(double kappa) { return -kappa * 1.4426950408889634; }
__device__ __forceinline__ ds exp_scale(ds kappa) { return -kappa * lit<ds>(1.4426950408889634); }
template <typename real>
__device__ __forceinline__ real exp2_scaled(real s, real r) {
    return exp2_(mul_(s, r));
}
// 1/sqrt of a squared distance formed with a cancellation: a value rounded
// below zero is taken by its magnitude (FP32; FP64 keeps 29 bits more)
__device__ __forceinline__ float rsqrt_abs(float x) { return rsqrt_fast(fabsf(x)); }
__device__ __forceinline__ double rsqrt_abs(double x) { return rsqrt_fast(x); }

// One panel staged for the P2P sums: the centroid relative to the group's
// centre (PanelGeo holds it relative to the leaf's), 2 (v_0 - c), 2 (v_1 - c),
// the unit normal, g_k = |v_k - c|^2, and the densities times the area:
// {psi_L, psi_Y, phi of the Laplace pair, phi}; the Laplace two are zero
// unless the panel and the group share a dielectric body.  sliver: not zero for
// a long thin panel (is_sliver).
template <typename real>
struct __align__(16) PanelS {
    real cx, cy, cz, g0;
    real ux, uy, uz, g1;
    real vx, vy, vz, g2;
    real nx, ny, nz, sliver;
    real qL, qY, pL, pY;
};

// The sums of panel_sums point by point, for slivers: every point's own offset
// e = d + a s_k, squared distance and normal product n.e (h is 1 then), 19
// FMA-pipe operations a point.  For a triangle of 10 by 0.05 and targets 0.01
// from its outer points the panel form is off by up to 3e-2 in FP32 and 9e-11 in
// FP64, this by what the coordinates leave, 7e-4 and 3e-12.  A stage of columns
// without a sliver does not ask for one: asking panel by panel cost the FP32
// product 4 %.
template <typename real, int K, bool LAP>
__device__ __forceinline__ void point_sums(const PanelS<real>& q, real X, real Y, real Z, real kappa, real nkl,
                                           const real (&ra)[2], const real (&rw)[3], real& VL, real& KL, real& VY,
                                           real& KY) {
    const real dx = X - q.cx, dy = Y - q.cy, dz = Z - q.cz;
    VL = KL = VY = KY = real(0);
#pragma unroll 1
    for (int m = K == 3 ? 1 : 0; m < (K == 3 ? 4 : K); ++m) {
        const int k = m > 3 ? m - 3 : m;  // vertex 1..3 of the orbit, 0: the centroid
        const real b = k == 0 ? real(0) : real(0.5) * (m > 3 ? ra[1] : ra[0]);
        const real w = m == 0 ? rw[0] : (m > 3 ? rw[2] : rw[1]);
        // b times 2 s_k; the third vertex's is minus the others' sum
        const real ex = fma_(b, k == 1 ? q.ux : (k == 2 ? q.vx : -(q.ux + q.vx)), dx);
        const real ey = fma_(b, k == 1 ? q.uy : (k == 2 ? q.vy : -(q.uy + q.vy)), dy);
        const real ez = fma_(b, k == 1 ? q.uz : (k == 2 ? q.vz : -(q.uz + q.vz)), dz);
        const real r2 = fma_(ez, ez, fma_(ey, ey, mul_(ex, ex)));
        const real h = fma_(q.nz, ez, fma_(q.ny, ey, mul_(q.nx, ex)));
        const real ri = rsqrt_abs(r2);
        const real t = mul_(h, mul_(ri, ri));
        const real r = mul_(r2, ri);
        const real e = mul_(w, mul_(exp2_scaled(nkl, r), ri));
        if (LAP) {
            const real v = mul_(w, ri);
            VL = add_(VL, v);
            KL = fma_(v, t, KL);
        }
        VY = add_(VY, e);
        KY = fma_(mul_(e, fma_(kappa, r, real(1))), t, KY);
    }
}

// Sums over the far rule's points of one panel for one target at X (relative
// to the group's centre).  The rule's points are c and c - 3 alpha s_k, s_k =
// v_k - c, so with d = X - c and a = 3 alpha
//   |X - y|^2 = |d|^2 + a (2 d.s_k + a |s_k|^2),
// two operations a point instead of six, and n.(X - y) = n.d is the panel's:
//   V = sum w / r, K = n.d sum w / r^3 (Laplace), with e^{-kappa r} and
//   (1 + kappa r) e^{-kappa r} for Yukawa; U += q V - p K.
// The densities and the normal product are met once per panel.  In FP32 a
// point costs 15 FMA-pipe operations with the panel's share (19 point by
// point) and 2 MUFU (16 cycles a warp), and a panel five 16-byte shared loads
// instead of 14.  The squared distance
// loses a factor |d|^2 / r^2 of relative accuracy, below ten on shape-regular
// panels, of the order of what the FP32 coordinates leave, and n.d rounds at
// the size of d instead of X - y; on slivers, whose points come close to targets
// far from the centroid, both show (point_sums).  (Double-single sums point by
// point throughout: p2p_ds.cuh.)
// panel_sums: V_L, sum w / r^3, V_Y and its counterpart (without n.d), and n.d.
// SLIVER: the panel may be one.
template <typename real, int K, bool LAP, bool SLIVER>
__device__ __forceinline__ void panel_sums(const PanelS<real>& q, real X, real Y, real Z, real kappa, real nkl,
                                           const real (&ra)[2], const real (&rw)[3], real& VL, real& KL, real& VY,
                                           real& KY, real& h) {
    if (SLIVER && q.sliver != real(0)) {  // (all lanes alike)
        point_sums<real, K, LAP>(q, X, Y, Z, kappa, nkl, ra, rw, VL, KL, VY, KY);
        h = real(1);
        return;
    }
    const real dx = X - q.cx, dy = Y - q.cy, dz = Z - q.cz;
    const real D2 = fma_(dz, dz, fma_(dy, dy, mul_(dx, dx)));
    h = fma_(q.nz, dz, fma_(q.ny, dy, mul_(q.nx, dx)));
    const real one = real(1);
    VL = KL = VY = KY = real(0);
    auto point = [&](const real r2, real& sV, real& sK, real& sW, real& sM, bool first) {
        const real ri = rsqrt_abs(r2);
        const real i2 = mul_(ri, ri);
        const real r = mul_(r2, ri);
        const real e = mul_(exp2_scaled(nkl, r), ri);
        const real gg = fma_(kappa, r, one);
        const real e2 = mul_(e, i2);
        if (first) {
            if (LAP) {
                sV = ri;
                sK = mul_(ri, i2);
            }
            sW = e;
            sM = mul_(e2, gg);
        } else {
            if (LAP) {
                sV = add_(sV, ri);
                sK = fma_(ri, i2, sK);
            }
            sW = add_(sW, e);
            sM = fma_(e2, gg, sM);
        }
    };
    if (K != 3) {
        real sV, sK, sW, sM;
        point(D2, sV, sK, sW, sM, true);
        if (LAP) {
            VL = mul_(rw[0], sV);
            KL = mul_(rw[0], sK);
        }
        VY = mul_(rw[0], sW);
        KY = mul_(rw[0], sM);
    }
    if (K >= 3) {
        const real p0 = fma_(q.uz, dz, fma_(q.uy, dy, mul_(q.ux, dx)));
        const real p1 = fma_(q.vz, dz, fma_(q.vy, dy, mul_(q.vx, dx)));
        const real p2 = -add_(p0, p1);
        if constexpr (std::is_same<real, float>::value && K == 7) {
            // the two orbits side by side as packed halves: with the stage's loop
            // kept rolled (63 registers, 32 warps an SM) the issue slots no longer
            // bound the sums: product of 2 x 20480 panels 202 -> 193 us, of 2 x
            // 204020 2143 -> 2061 us (packed but unrolled by the compiler: 199, 2106)
            const f2 a2{ra[0], ra[1]}, k2{kappa, kappa}, n2{nkl, nkl}, o2{1.f, 1.f};
            f2 tV, tK, tW, tM;
            auto both = [&](const float p, const float g, bool first) {
                const f2 r2 = fma_(a2, fma_(a2, f2{g, g}, f2{p, p}), f2{D2, D2});
                const f2 ri{rsqrt_abs(r2.a), rsqrt_abs(r2.b)};
                const f2 i2 = mul_(ri, ri);
                const f2 r = mul_(r2, ri);
                const f2 x = mul_(n2, r);
                const f2 e = mul_(f2{exp2_(x.a), exp2_(x.b)}, ri);
                const f2 gg = fma_(k2, r, o2);
                const f2 e2 = mul_(e, i2);
                if (first) {
                    if (LAP) {
                        tV = ri;
                        tK = mul_(ri, i2);
                    }
                    tW = e;
                    tM = mul_(e2, gg);
                } else {
                    if (LAP) {
                        tV = add_(tV, ri);
                        tK = fma_(ri, i2, tK);
                    }
                    tW = add_(tW, e);
                    tM = fma_(e2, gg, tM);
                }
            };
            both(p0, q.g0, true);
            both(p1, q.g1, false);
            both(p2, q.g2, false);
            if (LAP) {
                VL = fmaf(rw[1], tV.a, fmaf(rw[2], tV.b, VL));
                KL = fmaf(rw[1], tK.a, fmaf(rw[2], tK.b, KL));
            }
            VY = fmaf(rw[1], tW.a, fmaf(rw[2], tW.b, VY));
            KY = fmaf(rw[1], tM.a, fmaf(rw[2], tM.b, KY));
            return;
        }
#pragma unroll
        for (int o = 0; o < (K == 7 ? 2 : 1); ++o) {
            real sV, sK, sW, sM;
            point(fma_(ra[o], fma_(ra[o], q.g0, p0), D2), sV, sK, sW, sM, true);
            point(fma_(ra[o], fma_(ra[o], q.g1, p1), D2), sV, sK, sW, sM, false);
            point(fma_(ra[o], fma_(ra[o], q.g2, p2), D2), sV, sK, sW, sM, false);
            if (LAP) {
                VL = fma_(rw[1 + o], sV, VL);
                KL = fma_(rw[1 + o], sK, KL);
            }
            VY = fma_(rw[1 + o], sW, VY);
            KY = fma_(rw[1 + o], sM, KY);
        }
    }
}
template <typename real, int K, bool LAP, bool OWN, bool SLIVER>
__device__ __forceinline__ void p2p_panel(const PanelS<real>& q, bool own, real X, real Y, real Z, real kappa,
                                          real nkl, const real (&ra)[2], const real (&rw)[3], real& UL, real& UY) {
    real VL, KL, VY, KY, h;
    panel_sums<real, K, LAP, SLIVER>(q, X, Y, Z, kappa, nkl, ra, rw, VL, KL, VY, KY, h);
    if (OWN && own) VL = KL = VY = KY = real(0);  // the panel's own integral is a near-field correction
    if (LAP) UL = fma_(q.qL, VL, fma_(mul_(-q.pL, h), KL, UL));
    UY = fma_(q.qY, VY, fma_(mul_(-q.pY, h), KY, UY));
}

// Partial sums of the NW warps of a block combined in warp order (each warp
// carries a compensated pair per kernel) and stored per lane for the item.
template <typename real, int NW>
__device__ __forceinline__ void store_item(real (*red)[4][32], int w, int lane, real UL, real cL, real UY, real cY,
                                           double* out) {
    red[w][0][lane] = UL;
    red[w][1][lane] = cL;
    red[w][2][lane] = UY;
    red[w][3][lane] = cY;
    __syncthreads();
    if (w == 0) {
        real sL = 0, eL = 0, sY = 0, eY = 0;
        for (int k = 0; k < NW; ++k) {
            kadd(sL, eL, red[k][0][lane]);
            kadd(sL, eL, red[k][1][lane]);
            kadd(sY, eY, red[k][2][lane]);
            kadd(sY, eY, red[k][3][lane]);
        }
        out[lane] = to_dbl(sL) + to_dbl(eL);
        out[32 + lane] = to_dbl(sY) + to_dbl(eY);
    }
}

// Centroid of a column's panel relative to the group's centre: in FP32 from the
// column (one rounding of the FP64 difference), in FP64 the centroid
// relative to its leaf's centre plus the difference of the centres.
template <typename real>
__device__ __forceinline__ void col_centroid(const EvalArgs& a, const float4& c, int j, int64_t g,
                                             const real* __restrict__ v, real& x, real& y, real& z) {
    if constexpr (sizeof(real) == sizeof(float)) {
        x = c.x;
        y = c.y;
        z = c.z;
    } else {
        const int nd = a.pnode[j];
        x = v[0] + from_dbl<real>(a.ncenter[3 * nd] - a.gcenter[3 * g]);
        y = v[1] + from_dbl<real>(a.ncenter[3 * nd + 1] - a.gcenter[3 * g + 1]);
        z = v[2] + from_dbl<real>(a.ncenter[3 * nd + 2] - a.gcenter[3 * g + 2]);
    }
}

// The geometry of panel j (column c of group g) into q.
template <typename real, int K>
__device__ __forceinline__ void stage_panel(const EvalArgs& a, const float4& c, int j, int64_t g, PanelS<real>& q) {
    // the first 16 values of a staged panel, relative to the leaf
    const PanelS<real>& v = *reinterpret_cast<const PanelS<real>*>((const real*)a.pg + 16 * (int64_t)j);
    col_centroid<real>(a, c, j, g, &v.cx, q.cx, q.cy, q.cz);
    if (K > 1) {  // (one point: the centroid)
        q.g0 = v.g0;
        q.ux = v.ux;
        q.uy = v.uy;
        q.uz = v.uz;
        q.g1 = v.g1;
        q.vx = v.vx;
        q.vy = v.vy;
        q.vz = v.vz;
        q.g2 = v.g2;
        q.sliver = v.sliver;
    }
    q.nx = v.nx;
    q.ny = v.ny;
    q.nz = v.nz;
}

// Panels summed plainly before they join the compensated sums: about the 32
// points of rounding growth that the FP32 product's accuracy rests on.  (All
// 32 panels of a stage in one plain sum: 10-20 % more error against FP64.)
// With the one-point rule twice as many, unrolled: a panel is 17 operations
// there, and neither the loop nor the compensation is paid for by other points
// (direct sum of 2 x 20480 panels 2.17 -> 1.83 ms).
#define P2P_RUN 4

// P2P: one block of NW warps per work item, i.e. an even share of the columns
// (panels of the near leaves) of one target group (32 targets, one per lane).
// The item's columns go to the warps in NW even runs; a warp stages up to 32
// panels at a time, one per lane, moved to the group's frame, and every lane
// then sums them for its target (p2p_panel).  The panels of several leaves
// share a stage, so a warp's steps are full whatever the leaf sizes.  The
// item's partial sums go to Up.
//
// FP64 is compiled for two blocks on an SM (126 registers at seven points).
// Left to itself the compiler takes 80 registers and spills, three blocks fit,
// and they keep the upward pass and the M2P, which run beside them, out of the
// SMs: products of 4240 panels at order 8 1.50 -> 1.27 ms, of 4500 panels with
// the four-point rule 1.38 -> 1.21 ms.  Where the P2P is most of the product
// (order 6, seven points) 1.65 ms either way, and 1.67 -> 1.73 ms with the
// geometry out of cache.  (96 registers: 1.27, 1.27 and 1.69 ms.)  FP32 takes 63
// or 64 registers by itself; the bound would make it 91.
template <typename real, int K, int NW>
__global__ void __launch_bounds__(NW * 32, sizeof(real) == 8 ? 2 : 0) k_p2p(EvalArgs a, const typename V4<real>::t* __restrict__ xrel) {
    __shared__ __align__(16) PanelS<real> sP[NW][32];
    __shared__ real red[NW][4][32];
    __shared__ int64_t s_item;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned long long dm = body_mask(a.bmask), act = a.src_mask & dm;
    const real kappa = (real)a.kappa;
    const real nkl = exp_scale(kappa);
    const real ra[2] = {from_dbl<real>(a.rule.a[0]), from_dbl<real>(a.rule.a[1])};
    const real rw[3] = {from_dbl<real>(a.rule.w[0]), from_dbl<real>(a.rule.w[1]), from_dbl<real>(a.rule.w[2])};
    const real* __restrict__ pd = (const real*)a.pd;
    for (int64_t it = next_item(a.p2p_work, -1, &s_item); it < a.n_pitems; it = next_item(a.p2p_work, it, &s_item)) {
        const int64_t g = a.pitem_group[it];
        const int gb = a.gbody[g];
        if (!(((a.tgt_mask & dm) >> gb) & 1ull) || g < a.g_lo || g >= a.g_hi) continue;  // rows not used (block-uniform)
        const int p0 = a.gstart[g], p1 = a.gend[g];
        const int p = p0 + lane;
        const typename V4<real>::t xr = xrel[p < p1 ? p : p0];
        const real X = xr.x, Y = xr.y, Z = xr.z;
        const bool glap = a.lap_body[gb];
        real UL = 0, cL = 0, UY = 0, cY = 0;
        // the item's columns, then this warp's
        const int64_t i0 = a.pitem_off[g], c0 = a.col_off[g], nc = a.col_off[g + 1] - c0;
        const int64_t per = (nc + a.pitem_off[g + 1] - i0 - 1) / (a.pitem_off[g + 1] - i0);
        const int64_t b0 = c0 + (it - i0) * per, b1 = min(c0 + nc, b0 + per);
        const int64_t wper = b1 > b0 ? (b1 - b0 + NW - 1) / NW : 0;
        const int64_t w1 = min(b1, b0 + (w + 1) * wper);
        for (int64_t e = b0 + w * wper; e < w1; e += 32) {
            const int cnt = (int)min((int64_t)32, w1 - e);
            bool lap = false, has_own = false, sliver = false, on = false;
            int own = -1;  // the stage's slot of this lane's own panel
            int j = -1, b = 0;
            float4 c;
            if (lane < cnt) {
                c = column(a, g, c0, e - c0 + lane);
                j = __float_as_int(c.w);
                b = a.pbody[j];
                on = (act >> b) & 1ull;
            }
            // a body without density in this product adds nothing; a group's
            // columns ascend by body, so its stages are left out whole
            if (!__any_sync(0xffffffffu, on)) continue;
            __syncwarp();
            if (lane < cnt) {
                lap = glap && b == gb;
                has_own = j >= p0 && j < p1;
                PanelS<real>& q = sP[w][lane];
                stage_panel<real, K>(a, c, j, g, q);
                sliver = K >= 3 && q.sliver != real(0);
                const real z = real(0);
                q.qL = on && lap ? pd[4 * (int64_t)j] : z;
                q.qY = on ? pd[4 * (int64_t)j + 1] : z;
                const real ph = on ? pd[4 * (int64_t)j + 2] : z;
                q.pL = lap ? ph : z;
                q.pY = ph;
            }
            lap = __any_sync(0xffffffffu, lap);
            has_own = __any_sync(0xffffffffu, has_own);
            sliver = __any_sync(0xffffffffu, sliver);
            if (has_own)
                for (int k = 0; k < cnt; ++k)
                    if (__shfl_sync(0xffffffffu, j, k) == p) own = k;
            __syncwarp();
            // a few panels in plain sums, then into the compensated ones
            auto sums = [&](auto LAPc, auto OWNc, auto SLVc) {
                constexpr int RUN = K == 1 ? 2 * P2P_RUN : P2P_RUN;
                for (int k0 = 0; k0 < cnt; k0 += RUN) {
                    real sumL = 0, sumY = 0;
                    const int k1 = min(cnt, k0 + RUN);
#pragma unroll(K == 1 ? RUN : 1)
                    for (int k = k0; k < k1; ++k)
                        p2p_panel<real, K, decltype(LAPc)::value, decltype(OWNc)::value, decltype(SLVc)::value>(
                            sP[w][k], k == own, X, Y, Z, kappa, nkl, ra, rw, sumL, sumY);
                    if (decltype(LAPc)::value) kadd(UL, cL, sumL);
                    kadd(UY, cY, sumY);
                }
            };
            const std::true_type yes;
            const std::false_type no;
            if (sliver) {
                sums(yes, yes, yes);  // (the Laplace densities are zero where they do not apply)
            } else if (has_own) {
                if (lap) sums(yes, yes, no);
                else sums(no, yes, no);
            } else {
                if (lap) sums(yes, no, no);
                else sums(no, no, no);
            }
        }
        store_item<real, NW>(red, w, lane, UL, cL, UY, cY, a.Up + 64 * it);
    }
}

// ---------------------------------------------------------------- stored near field
// A GMRES solve applies the same near field tens of times, so it keeps the
// panel sums of every (target, column) pair: V_Y and K_Y = n.d sum.., and on a
// group's own dielectric body V_L and K_L before them (the own panel: zeros).
// A product then streams them, 16 or 8 bytes a pair in FP32, instead of
// forming seven points each.  Layout: per column units of 32 lanes x 2 values,
// two units {V_L, K_L}, {V_Y, K_Y} where the Laplace pair is kept (lane by lane
// four values in FP32), else one.  The Laplace columns of a group are one run.
struct NearGroup {
    int64_t unit;     // first unit of the group's columns
    int32_t l0, l1;   // its Laplace columns, counted from its first column
};
__host__ __device__ __forceinline__ int64_t near_unit(const NearGroup& n, int64_t c) {
    const int64_t in = c - n.l0;
    return n.unit + c + (in < 0 ? 0 : (in < n.l1 - n.l0 ? in : n.l1 - n.l0));
}
template <typename real, bool LAP>
__device__ __forceinline__ void near_store(real* u, int lane, real vl, real kl, real vy, real ky) {
    if constexpr (!LAP) {
        u[2 * lane] = vy;
        u[2 * lane + 1] = ky;
    } else if constexpr (sizeof(real) == 4) {
        reinterpret_cast<float4*>(u)[lane] = make_float4(vl, kl, vy, ky);
    } else {
        reinterpret_cast<double2*>(u)[lane] = make_double2(vl, kl);
        reinterpret_cast<double2*>(u)[32 + lane] = make_double2(vy, ky);
    }
}

// Forms the matrix: one block per P2P item, as k_p2p.
template <typename real, int K, int NW>
__global__ void __launch_bounds__(NW * 32) k_near_build(EvalArgs a, const NearGroup* __restrict__ ng,
                                                        const typename V4<real>::t* __restrict__ xrel,
                                                        real* __restrict__ mat) {
    __shared__ __align__(16) PanelS<real> sP[NW][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const real kappa = (real)a.kappa;
    const real nkl = exp_scale(kappa);
    const real ra[2] = {from_dbl<real>(a.rule.a[0]), from_dbl<real>(a.rule.a[1])};
    const real rw[3] = {from_dbl<real>(a.rule.w[0]), from_dbl<real>(a.rule.w[1]), from_dbl<real>(a.rule.w[2])};
    const int64_t it = blockIdx.x, g = a.pitem_group[it];
    const int p0 = a.gstart[g], p1 = a.gend[g];
    const int p = p0 + lane;
    const typename V4<real>::t xr = xrel[p < p1 ? p : p0];
    const NearGroup nm = ng[g];
    const int64_t i0 = a.pitem_off[g], c0 = a.col_off[g], nc = a.col_off[g + 1] - c0;
    const int64_t per = (nc + a.pitem_off[g + 1] - i0 - 1) / (a.pitem_off[g + 1] - i0);
    const int64_t b0 = (it - i0) * per, b1 = min(nc, b0 + per);
    const int64_t wper = b1 > b0 ? (b1 - b0 + NW - 1) / NW : 0;
    const int64_t w1 = min(b1, b0 + (w + 1) * wper);
    for (int64_t e = b0 + w * wper; e < w1; e += 32) {
        const int cnt = (int)min((int64_t)32, w1 - e);
        __syncwarp();
        int j = -1;
        if (lane < cnt) {
            const float4 c = a.col[c0 + e + lane];
            j = __float_as_int(c.w);
            stage_panel<real, K>(a, c, j, g, sP[w][lane]);
        }
        __syncwarp();
        for (int k = 0; k < cnt; ++k) {
            // zeros for the own panel and for lanes without a target
            const bool own = __shfl_sync(0xffffffffu, j, k) == p || p >= p1;
            const int64_t c = e + k;
            real* u = mat + 64 * near_unit(nm, c);
            real VL, KL, VY, KY, h;
            if (c >= nm.l0 && c < nm.l1) {
                panel_sums<real, K, true, (K >= 3)>(sP[w][k], xr.x, xr.y, xr.z, kappa, nkl, ra, rw, VL, KL, VY, KY, h);
                const real z = 0;
                near_store<real, true>(u, lane, own ? z : VL, own ? z : h * KL, own ? z : VY, own ? z : h * KY);
            } else {
                panel_sums<real, K, false, (K >= 3)>(sP[w][k], xr.x, xr.y, xr.z, kappa, nkl, ra, rw, VL, KL, VY, KY, h);
                const real z = 0;
                near_store<real, false>(u, lane, z, z, own ? z : VY, own ? z : h * KY);
            }
        }
    }
}

// The near-field sums of one product from the matrix, items and warps as in
// k_p2p; a warp keeps the densities of 32 columns in shared memory and eight
// columns' loads in flight.  Bound by HBM in FP32: 2 x 20480 panels hold 283 MB
// and take 56 us alone, 60 to 78 beside the upward pass (k_p2p: 101 us alone); by
// the FP64 pipe in FP64: 565 MB, 346 us (k_p2p: 9.3 ms).
template <typename real, int NW>
__global__ void __launch_bounds__(NW * 32) k_near(EvalArgs a, const NearGroup* __restrict__ ng,
                                                  const real* __restrict__ mat) {
    using v4 = typename V4<real>::t;
    constexpr int U = 8;
    __shared__ v4 sD[NW][32];  // psi_L, psi_Y, phi
    __shared__ real red[NW][4][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned long long dm = body_mask(a.bmask), act = a.src_mask & dm;
    const v4* __restrict__ pd = (const v4*)a.pd;
    const int64_t it = blockIdx.x, g = a.pitem_group[it];
    if (!(((a.tgt_mask & dm) >> a.gbody[g]) & 1ull)) return;  // rows not used (block-uniform)
    real UL = 0, cL = 0, UY = 0, cY = 0;
    const NearGroup nm = ng[g];
    const int64_t i0 = a.pitem_off[g], c0 = a.col_off[g], nc = a.col_off[g + 1] - c0;
    const int64_t per = (nc + a.pitem_off[g + 1] - i0 - 1) / (a.pitem_off[g + 1] - i0);
    const int64_t b0 = (it - i0) * per, b1 = min(nc, b0 + per);
    const int64_t wper = b1 > b0 ? (b1 - b0 + NW - 1) / NW : 0;
    const int64_t w1 = min(b1, b0 + (w + 1) * wper);
    for (int64_t e = b0 + w * wper; e < w1; e += 32) {
        const int cnt = (int)min((int64_t)32, w1 - e);
        __syncwarp();
        v4 d;
        d.x = d.y = d.z = d.w = 0;
        bool on = false;
        if (lane < cnt) {
            const int j = __float_as_int(a.col[c0 + e + lane].w);
            on = (act >> a.pbody[j]) & 1ull;
            if (on) d = pd[j];
        }
        if (!__any_sync(0xffffffffu, on)) continue;  // (as k_p2p)
        sD[w][lane] = d;
        __syncwarp();
        // runs of one kind of column
        for (int k = 0; k < cnt;) {
            const int64_t c = e + k;
            const bool lap = c >= nm.l0 && c < nm.l1;
            const int64_t lim = c < nm.l0 ? nm.l0 : (lap ? nm.l1 : nc);
            const int n = (int)min((int64_t)(cnt - k), lim - c);
            const real* u = mat + 64 * near_unit(nm, c);
            for (int q = 0; q < n; q += U) {
                real sL = 0, sY = 0;
                if (lap) {
                    real v[U][4];
#pragma unroll
                    for (int r = 0; r < U; ++r) {
                        const real* p = u + 128 * (int64_t)min(q + r, n - 1);
                        if constexpr (sizeof(real) == 4) {
                            const float4 x = __ldcs(reinterpret_cast<const float4*>(p) + lane);
                            v[r][0] = x.x;
                            v[r][1] = x.y;
                            v[r][2] = x.z;
                            v[r][3] = x.w;
                        } else {
                            const double2 x = __ldcs(reinterpret_cast<const double2*>(p) + lane);
                            const double2 y = __ldcs(reinterpret_cast<const double2*>(p) + 32 + lane);
                            v[r][0] = x.x;
                            v[r][1] = x.y;
                            v[r][2] = y.x;
                            v[r][3] = y.y;
                        }
                    }
#pragma unroll
                    for (int r = 0; r < U; ++r)
                        if (q + r < n) {
                            const v4 s = sD[w][k + q + r];
                            sL += v[r][0] * s.x - v[r][1] * s.z;
                            sY += v[r][2] * s.y - v[r][3] * s.z;
                        }
                } else {
                    real v[U][2];
#pragma unroll
                    for (int r = 0; r < U; ++r) {
                        const real* p = u + 64 * (int64_t)min(q + r, n - 1) + 2 * lane;
                        if constexpr (sizeof(real) == 4) {
                            const float2 x = __ldcs(reinterpret_cast<const float2*>(p));
                            v[r][0] = x.x;
                            v[r][1] = x.y;
                        } else {
                            const double2 x = __ldcs(reinterpret_cast<const double2*>(p));
                            v[r][0] = x.x;
                            v[r][1] = x.y;
                        }
                    }
#pragma unroll
                    for (int r = 0; r < U; ++r)
                        if (q + r < n) {
                            const v4 s = sD[w][k + q + r];
                            sY += v[r][0] * s.y - v[r][1] * s.z;
                        }
                }
                if (lap) kadd(UL, cL, sL);
                kadd(UY, cY, sY);
            }
            k += n;
        }
    }
    store_item<real, NW>(red, w, lane, UL, cL, UY, cY, a.Up + 64 * it);
}

template <typename real>
void launch_near_build(const EvalArgs& ev, int K, const void* ng, const void* xrel, void* mat, cudaStream_t s) {
    constexpr int NW = 8;
    using x4 = typename V4<real>::t;
    if (ev.n_pitems <= 0) return;
    const unsigned grid = (unsigned)ev.n_pitems;
    const NearGroup* n = (const NearGroup*)ng;
    switch (K) {
        case 1: k_near_build<real, 1, NW><<<grid, NW * 32, 0, s>>>(ev, n, (const x4*)xrel, (real*)mat); break;
        case 3: k_near_build<real, 3, NW><<<grid, NW * 32, 0, s>>>(ev, n, (const x4*)xrel, (real*)mat); break;
        case 4: k_near_build<real, 4, NW><<<grid, NW * 32, 0, s>>>(ev, n, (const x4*)xrel, (real*)mat); break;
        case 7: k_near_build<real, 7, NW><<<grid, NW * 32, 0, s>>>(ev, n, (const x4*)xrel, (real*)mat); break;
        default: fail(PGB_EINVAL, "K must be 1, 3, 4 or 7");
    }
}

// The P2P launch for the context's far rule.
template <typename real>
void launch_p2p(const EvalArgs& ev, int K, const void* xrel, cudaStream_t s) {
    constexpr int NW = 8;  // warps per block
    using x4 = typename V4<real>::t;
    if (ev.n_pitems <= 0) return;
    if (ev.near_mat) {
        k_near<real, NW><<<(unsigned)ev.n_pitems, NW * 32, 0, s>>>(ev, (const NearGroup*)ev.near_group,
                                                                   (const real*)ev.near_mat);
        return;
    }
    const unsigned grid = (unsigned)(ev.p2p_work ? ev.persist_blocks : ev.n_pitems);
    switch (K) {
        case 1: k_p2p<real, 1, NW><<<grid, NW * 32, 0, s>>>(ev, (const x4*)xrel); break;
        case 3: k_p2p<real, 3, NW><<<grid, NW * 32, 0, s>>>(ev, (const x4*)xrel); break;
        case 4: k_p2p<real, 4, NW><<<grid, NW * 32, 0, s>>>(ev, (const x4*)xrel); break;
        case 7: k_p2p<real, 7, NW><<<grid, NW * 32, 0, s>>>(ev, (const x4*)xrel); break;
        default: fail(PGB_EINVAL, "K must be 1, 3, 4 or 7");
    }
}

// M2P: one block of NW warps per work item, i.e. up to m2p_item far entries of
// one target group; the nodes go round robin to the warps, their far-field
// coefficients (k_far) staged in shared memory.  The item's partial sums go to
// Uf.  next_entry: the first entry from e on, in steps, whose source body is
// used in this product.
template <typename S>
__device__ __forceinline__ int64_t next_entry(const EvalArgs& a, int64_t e, int64_t f1, int step,
                                              unsigned long long dm) {
    if (a.all_active) return e;
    while (e < f1) {
        const int nd = sizeof(S) == sizeof(float) ? __float_as_int(a.far4[e].w) : a.far_l[e];
        const int b = a.nbody[nd];
        if (a.src_active[b] && ((dm >> b) & 1ull)) return e;
        e += step;
    }
    return e;
}

// FP32: a half warp takes a node, each of its 16 lanes two of the group's
// targets as the halves of packed values.  A target per lane in scalar
// arithmetic issued 384 instructions per (node, 32 targets) with monomials and
// 314 in the harmonic basis, at 56-64 % of the issue rate; packed, they halve
// (85 -> 65 us at order 6 for 2 x 20480 panels).  What is left is latency: 126
// registers hold 23 % of the warps, the issue slots are 53 % and the FMA pipe
// 31 % busy; fewer registers for more warps cost more than they gave (102: 1 %,
// 80: 3 % of the product).  The coefficients lie in shared memory twice over
// (c, c), ready as packed operands, and so do the recurrence constants.
template <int P, int NW>
__global__ void __launch_bounds__(NW * 32) k_m2p_f32(EvalArgs a, const float4* __restrict__ xrel,
                                                     const float* __restrict__ far) {
    constexpr int NC = n_far_pad(P), NV = 2 * NC / 4;  // 16-byte vectors of a node's coefficients
    constexpr int ML = (NV + 15) / 16;
    constexpr bool PRE = P <= 8;  // the next node's coefficients wait in registers
    __shared__ __align__(16) f2 sM[NW][2][2 * NC];
    __shared__ f2 sC[(P + 1) * (P + 1)];
    __shared__ float red[NW][4][32];
    __shared__ int64_t s_item;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, half = lane >> 4, hl = lane & 15;
    for (int k = threadIdx.x; k < (P + 1) * (P + 1); k += NW * 32) {
        const int l = k / (P + 1), m = k - l * (P + 1);
        const float c = l > 0 ? (float)(l * l - m * m) / (float)(4 * l * l - 1) : 0.f;
        sC[k] = f2{-c, -c};
    }
    __syncthreads();
    const unsigned long long dm = body_mask(a.bmask);
    const float4* __restrict__ farv = (const float4*)far;
    for (int64_t it = next_item(a.m2p_work, -1, &s_item); it < a.n_fitems; it = next_item(a.m2p_work, it, &s_item)) {
        const int64_t g = a.fitem_group[it];
        const int gb = a.gbody[g];
        if (!(((a.tgt_mask & dm) >> gb) & 1ull) || g < a.g_lo || g >= a.g_hi) continue;  // rows not used (block-uniform)
        const int64_t p0 = a.gstart[g], p1 = a.gend[g];
        const float4 xa = xrel[p0 + hl < p1 ? p0 + hl : p0], xb = xrel[p0 + 16 + hl < p1 ? p0 + 16 + hl : p0];
        const f2 kappa = cst<f2>(a.kappa);
        const bool glap = a.lap_body[gb];
        float UL[2] = {0, 0}, eL[2] = {0, 0}, UY[2] = {0, 0}, eY[2] = {0, 0};
        // the group's entries go evenly to its items
        const int64_t i0 = a.fitem_off[g], fo = a.far_off[g], nf = a.far_off[g + 1] - fo;
        const int64_t per = (nf + a.fitem_off[g + 1] - i0 - 1) / (a.fitem_off[g + 1] - i0);
        const int64_t fb = fo + (it - i0) * per, f1 = min(fo + nf, fb + per);
        int64_t e = next_entry<float>(a, fb + 2 * w + half, f1, 2 * NW, dm);
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f), pm[PRE ? ML : 1];
        int nb = -1;  // the node's body
        auto fetch = [&]() {
            if (e >= f1) return;
            q = a.far4[e];
            if (glap) nb = a.nbody[__float_as_int(q.w)];
            if constexpr (PRE) {
                const float4* c = farv + (int64_t)__float_as_int(q.w) * NV;
#pragma unroll
                for (int k = 0; k < ML; ++k)
                    if (hl + 16 * k < NV) pm[k] = c[hl + 16 * k];
            }
        };
        float4* sv = reinterpret_cast<float4*>(sM[w][half]);
        auto put = [&](int k, const float4& c) {
            sv[2 * k] = make_float4(c.x, c.x, c.y, c.y);
            sv[2 * k + 1] = make_float4(c.z, c.z, c.w, c.w);
        };
        fetch();
        while (__any_sync(0xffffffffu, e < f1)) {
            const bool on = e < f1;
            __syncwarp();
            if constexpr (PRE) {
#pragma unroll
                for (int k = 0; k < ML; ++k)
                    if (hl + 16 * k < NV) put(hl + 16 * k, pm[k]);
            } else if (on) {
                const float4* c = farv + (int64_t)__float_as_int(q.w) * NV;
                for (int k = hl; k < NV; k += 16) put(k, c[k]);
            }
            __syncwarp();
            const bool lap = on && glap && nb == gb;
            // a half without a node evaluates what its slots hold at a
            // harmless place and drops the result
            const f2 Rx = on ? f2{xa.x - q.x, xb.x - q.x} : f2{1.f, 1.f};
            const f2 Ry = on ? f2{xa.y - q.y, xb.y - q.y} : f2{0.f, 0.f};
            const f2 Rz = on ? f2{xa.z - q.z, xb.z - q.z} : f2{0.f, 0.f};
            if (on) e = next_entry<float>(a, e + 2 * NW, f1, 2 * NW, dm);
            fetch();  // the next node
            f2 uL, uY;
            if (__any_sync(0xffffffffu, lap)) {
                far_eval<f2, P, true>(Rx, Ry, Rz, kappa, sM[w][half], sM[w][half] + NC, sC, uL, uY);
                kadd(UL[0], eL[0], lap ? uL.a : 0.f);
                kadd(UL[1], eL[1], lap ? uL.b : 0.f);
            } else {
                far_eval<f2, P, false>(Rx, Ry, Rz, kappa, sM[w][half], sM[w][half] + NC, sC, uL, uY);
            }
            kadd(UY[0], eY[0], on ? uY.a : 0.f);
            kadd(UY[1], eY[1], on ? uY.b : 0.f);
        }
        // a lane keeps the target of its own number and gives the other half its other one
        const int give = 1 - half;
        const float oL = __shfl_xor_sync(0xffffffffu, give ? UL[1] : UL[0], 16);
        const float oeL = __shfl_xor_sync(0xffffffffu, give ? eL[1] : eL[0], 16);
        const float oY = __shfl_xor_sync(0xffffffffu, give ? UY[1] : UY[0], 16);
        const float oeY = __shfl_xor_sync(0xffffffffu, give ? eY[1] : eY[0], 16);
        float sL = half ? UL[1] : UL[0], cL = half ? eL[1] : eL[0], sY = half ? UY[1] : UY[0], cY = half ? eY[1] : eY[0];
        kadd(sL, cL, oL);
        kadd(sY, cY, oY);
        store_item<float, NW>(red, w, lane, sL, cL + oeL, sY, cY + oeY, a.Uf + 64 * it);
    }
}

// FP64 and double-single: a node per warp and a target per lane (bound by the
// FP64 and the FMA pipe; the shared loads hide behind them).
template <typename real, int P, int NW>
__global__ void __launch_bounds__(NW * 32) k_m2p(EvalArgs a,
                                                 const typename V4<typename Store<real>::S>::t* __restrict__ xrel,
                                                 const real* __restrict__ far) {
    using S = typename Store<real>::S;  // storage type of the targets
    using s4 = typename V4<S>::t;
    constexpr int NC = n_far_pad(P);
    extern __shared__ __align__(16) unsigned char m2p_smem[];
    real* sM = reinterpret_cast<real*>(m2p_smem) + (threadIdx.x >> 5) * 2 * NC;  // this warp's node
    float4* rad = reinterpret_cast<float4*>(m2p_smem + (size_t)NW * 2 * NC * sizeof(real)) + threadIdx.x;
    __shared__ real red[NW][4][32];
    __shared__ int64_t s_item;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned long long dm = body_mask(a.bmask);
    for (int64_t it = next_item(a.m2p_work, -1, &s_item); it < a.n_fitems; it = next_item(a.m2p_work, it, &s_item)) {
        const int64_t g = a.fitem_group[it];
        const int gb = a.gbody[g];
        if (!(((a.tgt_mask & dm) >> gb) & 1ull) || g < a.g_lo || g >= a.g_hi) continue;  // rows not used (block-uniform)
        const int64_t p0 = a.gstart[g], p1 = a.gend[g];
        const int64_t p = p0 + lane;
        const s4 xr = xrel[p < p1 ? p : p0];
        const double gc0 = a.gcenter[3 * g], gc1 = a.gcenter[3 * g + 1], gc2 = a.gcenter[3 * g + 2];
        const real kappa = to_c<real>((S)a.kappa);
        real UL = 0, cL = 0, UY = 0, cY = 0;
        // the group's entries go evenly to its items
        const int64_t i0 = a.fitem_off[g], fo = a.far_off[g], nf = a.far_off[g + 1] - fo;
        const int64_t per = (nf + a.fitem_off[g + 1] - i0 - 1) / (a.fitem_off[g + 1] - i0);
        const int64_t fb = fo + (it - i0) * per, f1 = min(fo + nf, fb + per);
        for (int64_t e = next_entry<S>(a, fb + w, f1, NW, dm); e < f1; e = next_entry<S>(a, e + NW, f1, NW, dm)) {
            const int nd = a.far_l[e];
            __syncwarp();
            for (int k = lane; k < 2 * NC; k += 32) sM[k] = far[(int64_t)nd * 2 * NC + k];
            __syncwarp();
            const bool lap = (a.nbody[nd] == gb) && a.lap_body[gb];
            const real Rx = to_c<real>(xr.x - (a.ncenter[3 * nd] - gc0));
            const real Ry = to_c<real>(xr.y - (a.ncenter[3 * nd + 1] - gc1));
            const real Rz = to_c<real>(xr.z - (a.ncenter[3 * nd + 2] - gc2));
            real uL, uY;
            if constexpr (is_ds<real>) {
                if (lap) far_eval_ds<P, true>(Rx, Ry, Rz, kappa, sM, sM + NC, rad, NW * 32, uL, uY);
                else far_eval_ds<P, false>(Rx, Ry, Rz, kappa, sM, sM + NC, rad, NW * 32, uL, uY);
            } else {
                if (lap) far_eval<real, P, true>(Rx, Ry, Rz, kappa, sM, sM + NC, nullptr, uL, uY);
                else far_eval<real, P, false>(Rx, Ry, Rz, kappa, sM, sM + NC, nullptr, uL, uY);
            }
            if (lap) kadd(UL, cL, uL);
            kadd(UY, cY, uY);
        }
        store_item<real, NW>(red, w, lane, UL, cL, UY, cY, a.Uf + 64 * it);
    }
}

struct UpArgs {
    int64_t n_leaves;
    const int32_t *leaf_node, *nstart, *nend, *child, *nchild, *nbody;
    int src_active[PGB_MAX_BODIES];
    const unsigned long long* bmask = nullptr;  // as EvalArgs::bmask
    const double* ncenter;
    int K;
    int sms;                     // the device's multiprocessors
    int p2m_grid;                // > 0: P2M over at most this many blocks (leaves strided)
    int64_t n_nodes;             // k_far: every node
    const void* far_tab;         // its table (farfield.cu) in the arithmetic type
    void* far;                   // its output: 2 * n_far_pad(P) coefficients per node
    FarRule rule;                // far rule (panel moments)
    const void* pg;              // panel geometry (PanelGeo) in the arithmetic type
    const void* pd;              // panel densities x area
    const void* pmom;            // panel moments (k_panel_moments), nullptr: formed in the P2M
    const int32_t* parent;       // k_climb: parent of every node (-1 at a body's root)
    int* arrive;                 // k_climb: per node, internal children finished (zero between launches)
    int64_t n_internal;          // k_climb: the nodes with children, in any order, and per node its
    const int32_t *internal_node, *n_ichild;  // children that have children
};
// a source body of the upward pass is used (its densities are not all zero
// and the run-time mask keeps it)
__device__ __forceinline__ bool body_on(const UpArgs& a, int b) {
    return a.src_active[b] && (!a.bmask || ((*a.bmask >> b) & 1ull));
}

// Far-field coefficients of every node of an active body from its moments
// (the tables of farfield.cu): a block takes NB nodes, whose moments it stages
// side by side in shared memory, and a thread forms one column of the Yukawa
// or the Laplace table for all of them, so that a table entry (coalesced, from
// L1 / L2) and NB / 4 shared loads serve NB multiply-adds.  Columns are
// ordered by degree, and a warp skips the moment degrees that none of its
// columns takes.  Output per node: Laplace then Yukawa coefficients in the
// order of far_pos.
template <typename real, int P, int NB>
__global__ void __launch_bounds__(2 * far_cols(P)) k_far(UpArgs a, const real* __restrict__ mom) {
    constexpr int T = MI<P>::T, TR = far_cols(P), NC = n_far_pad(P);
    constexpr int U = 8;  // table entries in flight per thread
    extern __shared__ __align__(16) unsigned char far_smem[];
    real(*sm)[NB] = reinterpret_cast<real(*)[NB]>(far_smem);  // [2 T][NB]
    const bool yuk = threadIdx.x < TR;
    const int j = yuk ? threadIdx.x : threadIdx.x - TR;
    const real* __restrict__ tab = (const real*)a.far_tab + (yuk ? 0 : (size_t)T * TR) + j;
    real* __restrict__ far = (real*)a.far;
    int l = 0;
    while ((l + 1) * (l + 1) <= j) ++l;
    const int r = j - l * l;
    const int m = (r + 1) / 2;
    const int out = (yuk ? NC : 0) + far_pos(P, l, m, r ? (r - 1) & 1 : 0);
    for (int64_t n0 = (int64_t)blockIdx.x * NB; n0 < a.n_nodes; n0 += (int64_t)gridDim.x * NB) {
        const int nn = (int)min((int64_t)NB, a.n_nodes - n0);
        bool act[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) act[i] = i < nn && body_on(a, a.nbody[n0 + i]);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < NB; ++i)
            for (int k = threadIdx.x; k < 2 * T; k += blockDim.x)
                sm[k][i] = act[i] ? mom[(n0 + i) * 2 * T + k] : real(0);
        __syncthreads();
        real acc[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) acc[i] = real(0);
        const real(*sk)[NB] = yuk ? sm + T : sm;
#pragma unroll 1
        for (int q = 0; q <= P; ++q) {
            const bool takes = l <= P && (yuk ? q >= l && !((q - l) & 1) : q == l);
            if (!__any_sync(0xffffffffu, takes)) continue;
            const int k0 = q * (q + 1) * (q + 2) / 6, k1 = k0 + (q + 1) * (q + 2) / 2;
#pragma unroll 1
            for (int k = k0; k < k1; k += U) {  // whole batches of loads, the last one masked
                real v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = k + u < k1 ? tab[(size_t)(k + u) * TR] : real(0);  // zero off the pattern
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int kk = min(k + u, k1 - 1);
#pragma unroll
                    for (int i = 0; i < NB; ++i) acc[i] = madd(v[u], sk[kk][i], acc[i]);
                }
            }
        }
        if (j < n_far(P))
#pragma unroll
            for (int i = 0; i < NB; ++i)
                if (act[i]) far[(n0 + i) * 2 * NC + out] = acc[i];
    }
}

// ---------------------------------------------------------------- upward pass
// P2M: a block per leaf (k_p2m).  Moment shifts in one launch (k_climb): a block
// per internal node whose children are all leaves; a node above runs in the
// block whose internal child finished last (a counter per node; the last of
// its internal children's increments goes on up, the others stop), so the tree
// is climbed without a launch or a barrier per level and no block waits for
// another.  Writers fence before their increment; the climbing block fences
// after it and reads the children's moments from L2 (ld.global.cg).  The
// far-field coefficients follow in k_far.  The whole pass is a chain of loads
// (its arithmetic is a few microseconds of the GPU): small blocks, many of
// them resident, and few steps in the chain are what it wants.  P2M and shifts
// in one kernel of 256-thread blocks held four blocks an SM, 65 us for 2968
// leaves.
//
// P2M.  The densities are constant on a panel, so with the panel's moments
// V_k = sum_m w_m u_m^k (the far rule's points, u = leaf centre - y) the leaf's
// moments are
//   M_k = sum_j A_j psi_j V_jk + sum_a k_a D_a[k - e_a],
//   D_a[k'] = sum_j A_j phi_j n_j,a V_jk':
// five multiply-adds per panel and k.  The V depend on the geometry alone; they
// are formed once per geometry (k_panel_moments) and read back coalesced.
#define UP_THREADS 256
// warps per child in k_climb: one up to order 8 (28 lines an axis at order 6),
// above (136 lines at order 15) four, two in the 8-byte types for their registers
__host__ __device__ constexpr int climb_wpc(int P, int bytes) { return P > 8 ? (bytes == 4 ? 4 : 2) : 1; }
__host__ __device__ __forceinline__ int mi_index(int x, int y, int z) {  // position in MI's order
    const int n = x + y + z;
    return n * (n + 1) * (n + 2) / 6 + (n - x) * (n - x + 1) / 2 + z;
}
constexpr int UP_CHUNK = 64;  // panels whose densities are staged at once
constexpr int UP_FLY = 4;     // panels whose point powers are staged at once (V formed on the spot)
// threads of a P2M block: one per multi-index, between 64 and 256
__host__ __device__ constexpr int p2m_threads(int P) {
    return n_terms(P) >= 256 ? 256 : (n_terms(P) <= 64 ? 64 : (n_terms(P) + 31) & ~31);
}
// Its threads take a leaf's panels in p2m_shares shares: thread tid those of its
// share p2m_share, and of each panel the moments of the multi-indices p2m_index
// (h = 0, 1, ..), -1 where it has none: the block is whole warps, so threads are
// left over at most orders (96 for the 84 multi-indices of order 6), and what
// they would read lies behind the last panel's moments.
__host__ __device__ constexpr int p2m_shares(int P) {
    return n_terms(P) >= p2m_threads(P) ? 1 : p2m_threads(P) / n_terms(P);
}
__host__ __device__ constexpr int p2m_share(int P, int tid) { return p2m_shares(P) > 1 ? tid / n_terms(P) : 0; }
__host__ __device__ constexpr int p2m_index(int P, int tid, int h) {
    const int k = tid - p2m_share(P, tid) * n_terms(P) + h * p2m_threads(P);
    return p2m_share(P, tid) < p2m_shares(P) && k < n_terms(P) ? k : -1;
}
template <typename real, int P, bool STORED>
struct P2MShared {
    static constexpr int T = MI<P>::T, BT = p2m_threads(P);
    static constexpr int NP = p2m_shares(P);         // shares of a leaf's panels
    real q[UP_CHUNK][5];                             // psi_L, psi_Y, phi n (all x area)
    real sum[NP][5][T];
    real pw[STORED ? 1 : UP_FLY * 7][3][P + 1];
    signed char kk[T][3];
};
template <typename real, int P>
struct ClimbShared {
    real buf[8][2 * MI<P>::T];
    real d[8][3];
    signed char ln[(P + 1) * (P + 2) / 2][2];
    int next;
};

template <typename real>
__device__ __forceinline__ real ld_cg(const real* p) {
    return __ldcg(p);
}
__device__ __forceinline__ ds ld_cg(const ds* p) {
    const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
    return ds(v.x, v.y);
}

// Powers of u = leaf centre - y at the far rule's points of panels j0 .. j0 + np - 1.
template <typename real, int P>
__device__ __forceinline__ void stage_powers(const UpArgs& a, int64_t j0, int np, real (*pw)[3][P + 1]) {
    for (int q = threadIdx.x; q < np * a.K * 3; q += blockDim.x) {
        const int pt = q / 3, ax = q - 3 * pt;
        const int jj = pt / a.K;
        const real* g = (const real*)a.pg + 16 * (j0 + jj);
        int m = pt - jj * a.K;
        real v = -g[ax];
        if (a.K != 3) --m;  // the centroid is point 0
        if (m >= 0) {
            const int o = m / 3, k = m - 3 * o;
            const real s0 = g[4 + ax], s1 = g[8 + ax];  // 2 (v_k - c); the third is minus their sum
            const real s = k == 0 ? s0 : (k == 1 ? s1 : -(s0 + s1));
            v = madd(from_dbl<real>(0.5 * a.rule.a[o]), s, v);  // y = c - 3 alpha s_k
        }
        real x = real(1);
#pragma unroll
        for (int d = 0; d <= P; ++d) {
            pw[pt][ax][d] = x;
            x = x * v;
        }
    }
}
// V_k of the staged panel whose points start at pw.
template <typename real, int P>
__device__ __forceinline__ real panel_moment(const UpArgs& a, const real (*pw)[3][P + 1], int kx, int ky, int kz) {
    real s = real(0);
    for (int m = 0; m < a.K; ++m) {
        const int o = a.K == 3 ? 1 : (m + 2) / 3;  // weight: centroid, first, second orbit
        s = madd(from_dbl<real>(a.rule.w[o]), (pw[m][0][kx] * pw[m][1][ky]) * pw[m][2][kz], s);
    }
    return s;
}

// The panel moments of all panels: out[j T + k].
template <typename real, int P>
__global__ void __launch_bounds__(UP_THREADS) k_panel_moments(UpArgs a, int64_t n_pan, real* __restrict__ out) {
    constexpr int T = MI<P>::T;
    __shared__ real pw[UP_FLY * 7][3][P + 1];
    __shared__ signed char kk[T][3];
    for (int k = threadIdx.x; k < T; k += blockDim.x) {
        int x, y, z;
        decode_mi(k, x, y, z);
        kk[k][0] = (signed char)x;
        kk[k][1] = (signed char)y;
        kk[k][2] = (signed char)z;
    }
    for (int64_t j0 = (int64_t)blockIdx.x * UP_FLY; j0 < n_pan; j0 += (int64_t)gridDim.x * UP_FLY) {
        const int np = (int)min((int64_t)UP_FLY, n_pan - j0);
        __syncthreads();
        stage_powers<real, P>(a, j0, np, pw);
        __syncthreads();
        for (int q = threadIdx.x; q < np * T; q += blockDim.x) {
            const int jj = q / T, k = q - jj * T;
            out[(j0 + jj) * T + k] = panel_moment<real, P>(a, pw + jj * a.K, kk[k][0], kk[k][1], kk[k][2]);
        }
    }
}

// P2M of a leaf into mom: a thread per multi-index, the panels in NP shares
// where T leaves threads over.
template <typename real, int P, bool STORED>
__global__ void __launch_bounds__(p2m_threads(P)) k_p2m(UpArgs a, real* __restrict__ mom) {
    using SH = P2MShared<real, P, STORED>;
    constexpr int T = SH::T, NP = SH::NP, BT = SH::BT;
    constexpr int H = (T + BT - 1) / BT;  // multi-indices per thread
    extern __shared__ __align__(16) unsigned char p2m_smem[];
    SH& sh = *reinterpret_cast<SH*>(p2m_smem);
    const int tid = threadIdx.x;
    const int part = p2m_share(P, tid), k0 = p2m_index(P, tid, 0);
    const bool on = k0 >= 0;
    for (int k = tid; k < T; k += BT) {
        int x, y, z;
        decode_mi(k, x, y, z);
        sh.kk[k][0] = (signed char)x;
        sh.kk[k][1] = (signed char)y;
        sh.kk[k][2] = (signed char)z;
    }
    for (int64_t leaf = blockIdx.x; leaf < a.n_leaves; leaf += gridDim.x) {
    const int nd = a.leaf_node[leaf];
    if (!body_on(a, a.nbody[nd])) continue;  // block-uniform
    const int64_t j0 = a.nstart[nd], j1 = a.nend[nd];
    const real* __restrict__ pg = (const real*)a.pg;
    const real* __restrict__ pd = (const real*)a.pd;
    const real* __restrict__ pm = (const real*)a.pmom;
    real acc[H][5];
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
        for (int c = 0; c < 5; ++c) acc[h][c] = real(0);
    auto add = [&](int h, real v, const real (&q)[5]) {
#pragma unroll
        for (int c = 0; c < 5; ++c) acc[h][c] = madd(v, q[c], acc[h][c]);
    };
    for (int64_t c0 = j0; c0 < j1; c0 += UP_CHUNK) {
        const int cnt = (int)min((int64_t)UP_CHUNK, j1 - c0);
        __syncthreads();
        if (tid < cnt) {
            const real* d = pd + 4 * (c0 + tid);
            const real* g = pg + 16 * (c0 + tid) + 12;
            sh.q[tid][0] = d[0];
            sh.q[tid][1] = d[1];
            for (int c = 0; c < 3; ++c) sh.q[tid][2 + c] = d[2] * g[c];
        }
        __syncthreads();
        if constexpr (STORED) {
            // all of a panel's moments at once: 8 to 16 loads in flight per thread
            if (on) {
                const real* v = pm + c0 * T + k0;
#pragma unroll(H >= 4 ? 4 : 8 / H)
                for (int j = part; j < cnt; j += NP) {
#pragma unroll
                    for (int h = 0; h < H; ++h)
                        if (h == 0 || p2m_index(P, tid, h) >= 0) add(h, v[(int64_t)j * T + h * BT], sh.q[j]);
                }
            }
        } else {
            for (int f = 0; f < cnt; f += UP_FLY) {
                const int np = min(UP_FLY, cnt - f);
                __syncthreads();
                stage_powers<real, P>(a, c0 + f, np, sh.pw);
                __syncthreads();
                if (on && part == 0)
#pragma unroll
                    for (int h = 0; h < H; ++h) {
                        const int k = p2m_index(P, tid, h);
                        if (k < 0) break;
                        for (int j = 0; j < np; ++j)
                            add(h, panel_moment<real, P>(a, sh.pw + j * a.K, sh.kk[k][0], sh.kk[k][1], sh.kk[k][2]),
                                sh.q[f + j]);
                    }
            }
        }
    }
    __syncthreads();
    if (on)
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const int k = p2m_index(P, tid, h);
            if (k >= 0)
#pragma unroll
                for (int c = 0; c < 5; ++c) sh.sum[part][c][k] = acc[h][c];
        }
    __syncthreads();
    auto total = [&](int c, int k) {
        real s = sh.sum[0][c][k];
#pragma unroll
        for (int p = 1; p < NP; ++p) s = s + sh.sum[p][c][k];
        return s;
    };
    for (int k = tid; k < T; k += BT) {
        const int x = sh.kk[k][0], y = sh.kk[k][1], z = sh.kk[k][2];
        real dl = real(0);
        if (x) dl = madd(real(x), total(2, mi_index(x - 1, y, z)), dl);
        if (y) dl = madd(real(y), total(3, mi_index(x, y - 1, z)), dl);
        if (z) dl = madd(real(z), total(4, mi_index(x, y, z - 1)), dl);
        mom[(int64_t)nd * 2 * T + k] = total(0, k) + dl;
        mom[(int64_t)nd * 2 * T + T + k] = total(1, k) + dl;
    }
    }
}

// Moment shift of node nd from its (at most eight) children,
// M_k(c) = sum_{j<=k} C(k,j) (c - c_child)^{k-j} M_j(c_child), climb_wpc warps
// per child: the shift is separable, and along an axis each line of moments
// s_0..s_n (the other two indices fixed) goes to a lane, which applies
// s_k += d s_{k-1}, k = n..t, for t = 1..n in registers (Pascal's triangle: after
// it s_k = sum_j C(k,j) d^{k-j} s_j), the Laplace and the Yukawa moments side by
// side (in FP32 as packed halves) -- no index tables, no binomials and no
// block barriers between the axes.  The children's sums follow in child order.
template <typename real>
struct PairOf {
    struct type {
        real a, b;
    };
};
template <>
struct PairOf<float> {
    using type = f2;
};
template <typename real>
using Pair = typename PairOf<real>::type;
__device__ __forceinline__ f2 pair_fma(f2 x, f2 y, f2 z) { return fma_(x, y, z); }
template <typename V>
__device__ __forceinline__ V pair_fma(const V& x, const V& y, const V& z) {
    return V{madd(x.a, y.a, z.a), madd(x.b, y.b, z.b)};
}
template <typename real, int P>
__device__ __forceinline__ void up_m2m(const UpArgs& a, int nd, int nc, int fc, real* __restrict__ mom,
                                       ClimbShared<real, P>& sh) {
    constexpr int T = MI<P>::T, NL = (P + 1) * (P + 2) / 2;  // lines per axis and kernel
    constexpr int CW = 32 * climb_wpc(P, sizeof(real));                     // threads per child
    const int tid = threadIdx.x, w = tid / CW, lane = tid - w * CW;
    // the threads of child w (a barrier of their own where they are several warps)
    auto sync_child = [&]() {
        if constexpr (CW == 32) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(w + 1), "n"(CW) : "memory");
    };
    __syncthreads();
    if (w < nc) {
        real* b = sh.buf[w];
        for (int k = lane; k < 2 * T; k += CW) b[k] = ld_cg(mom + (int64_t)(fc + w) * 2 * T + k);
        if (lane < 3) sh.d[w][lane] = from_dbl<real>(a.ncenter[3 * nd + lane] - a.ncenter[3 * (fc + w) + lane]);
        sync_child();
#pragma unroll 1
        for (int ax = 0; ax < 3; ++ax) {
            const Pair<real> dd{sh.d[w][ax], sh.d[w][ax]};
#pragma unroll 1
            for (int i = lane; i < (NL + CW - 1) / CW * CW; i += CW) {
                // the longest lines first: the lanes of a round have lines of
                // about one length, and the steps beyond the longest are left out
                const int li = min(i, NL - 1);
                const int e = sh.ln[li][0], f = sh.ln[li][1], n = i < NL ? P - e - f : -1;
                const int nm = __reduce_max_sync(0xffffffffu, n);
                Pair<real> s[P + 1];
                int at[P + 1];
#pragma unroll
                for (int k = 0; k <= P; ++k) {
                    at[k] = ax == 0 ? mi_index(k, e, f) : (ax == 1 ? mi_index(e, k, f) : mi_index(e, f, k));
                    s[k] = k <= n ? Pair<real>{b[at[k]], b[T + at[k]]} : Pair<real>{real(0), real(0)};
                }
#pragma unroll
                for (int t = 1; t <= P; ++t) {
                    if (t <= nm) {
#pragma unroll
                        for (int k = P; k >= t; --k)
                            if (k <= nm) s[k] = pair_fma(dd, s[k - 1], s[k]);
                    }
                }
#pragma unroll
                for (int k = 1; k <= P; ++k)
                    if (k <= n) {
                        b[at[k]] = s[k].a;
                        b[T + at[k]] = s[k].b;
                    }
            }
            sync_child();
        }
    }
    __syncthreads();
    for (int k = tid; k < 2 * T; k += blockDim.x) {
        real s = sh.buf[0][k];
        for (int c = 1; c < nc; ++c) s = s + sh.buf[c][k];
        mom[(int64_t)nd * 2 * T + k] = s;
    }
}

template <typename real, int P>
__global__ void __launch_bounds__(256 * climb_wpc(P, sizeof(real))) k_climb(UpArgs a, real* __restrict__ mom) {
    extern __shared__ __align__(16) unsigned char climb_smem[];
    ClimbShared<real, P>& sh = *reinterpret_cast<ClimbShared<real, P>*>(climb_smem);
    const int tid = threadIdx.x;
    bool ready = false;  // the line table is made when a node is shifted
    for (int64_t i = blockIdx.x; i < a.n_internal; i += gridDim.x) {
        int nd = a.internal_node[i];
        if (a.n_ichild[nd] > 0 || !body_on(a, a.nbody[nd])) continue;  // block-uniform
        if (!ready) {
            for (int q = tid; q < (P + 1) * (P + 2) / 2; q += blockDim.x) {  // (e, f) by e + f = 0..P
                int s = 0, r = q;
                while (r > s) r -= ++s;
                sh.ln[q][0] = (signed char)r;
                sh.ln[q][1] = (signed char)(s - r);
            }
            ready = true;  // (a barrier follows in up_m2m)
        }
        int nc = a.nchild[nd], fc = a.child[nd];
        for (;;) {
            // the parent's entries are fetched while nd is shifted
            const int par = a.parent[nd];
            int pic = 0, pnc = 0, pfc = 0;
            if (par >= 0) {
                pic = a.n_ichild[par];
                pnc = a.nchild[par];
                pfc = a.child[par];
            }
            up_m2m<real, P>(a, nd, nc, fc, mom, sh);
            // publish nd's moments, then count it at its parent
            __threadfence();
            __syncthreads();
            if (tid == 0) sh.next = par >= 0 && atomicAdd(a.arrive + par, 1) == pic - 1;
            __syncthreads();
            if (!sh.next) break;
            __threadfence();
            if (tid == 0) a.arrive[par] = 0;  // every internal child has arrived: ready for the next launch
            nd = par;
            nc = pnc;
            fc = pfc;
        }
    }
}

// M2P launch: blocks of 4 warps.
template <typename real, int P>
void launch_m2p(const EvalArgs& ev, const void* xrel, const void* far, cudaStream_t s) {
    if (ev.n_fitems <= 0) return;
    const unsigned grid = (unsigned)(ev.m2p_work ? ev.persist_blocks : ev.n_fitems);
    if constexpr (sizeof(real) == sizeof(float)) {
        constexpr int NW = 4;
        k_m2p_f32<P, NW><<<grid, NW * 32, 0, s>>>(ev, (const float4*)xrel, (const float*)far);
    } else {
        constexpr int NW = 4;
        constexpr size_t smem =
            NW * 2 * n_far_pad(P) * sizeof(real) + (is_ds<real> ? sizeof(float4) * NW * 32 * (P + 1) : 0);
        if constexpr (smem > 40 * 1024)
            PGB_CUDA(cudaFuncSetAttribute(k_m2p<real, P, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        k_m2p<real, P, NW><<<grid, NW * 32, smem, s>>>(
            ev, (const typename V4<typename Store<real>::S>::t*)xrel, (const real*)far);
    }
}

// The far-field coefficients: 8 nodes per block in FP32 and 4 in the 8-byte
// types (shared memory), where that gives every SM eight blocks; with fewer
// nodes, two and one per block, whose chain of loads is shorter (130 nodes:
// 8 us less for the whole product).  Above order 8 a block reads half a
// megabyte of table: half as many (658 nodes at order 15 make 165 blocks).
template <typename real, int P, int NB>
void launch_far_nb(const UpArgs& up, const void* mom, cudaStream_t s) {
    constexpr size_t smem = sizeof(real) * NB * 2 * MI<P>::T;
    if constexpr (smem > 40 * 1024)
        PGB_CUDA(cudaFuncSetAttribute(k_far<real, P, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int64_t gf = (up.n_nodes + NB - 1) / NB;
    if (up.p2m_grid > 0) gf = std::min<int64_t>(gf, up.p2m_grid);
    k_far<real, P, NB><<<(unsigned)std::max<int64_t>(gf, 1), 2 * far_cols(P), smem, s>>>(up, (const real*)mom);
}
template <typename real, int P>
void launch_far(const UpArgs& up, const void* mom, cudaStream_t s) {
    constexpr int NB = sizeof(real) == sizeof(float) ? 8 : 4;
    if (P > 8) launch_far_nb<real, P, NB / 2>(up, mom, s);
    else if (up.n_nodes >= (int64_t)8 * up.sms * NB) launch_far_nb<real, P, NB>(up, mom, s);
    else launch_far_nb<real, P, NB / 4>(up, mom, s);
}

// The panel moments of the current geometry (UpArgs::pg, rule, K) into out.
template <typename real, int P>
void launch_panel_moments(const UpArgs& up, int64_t n_pan, void* out, cudaStream_t s) {
    const int64_t grid = std::min<int64_t>((n_pan + UP_FLY - 1) / UP_FLY, (int64_t)8 * up.sms);
    if (grid > 0) k_panel_moments<real, P><<<(unsigned)grid, UP_THREADS, 0, s>>>(up, n_pan, (real*)out);
}

// The upward pass of one product: P2M, the moment shifts, the far-field
// coefficients.
template <typename real, int P>
void launch_upward(const UpArgs& up, void* mom, cudaStream_t s) {
    if (up.n_leaves <= 0) return;
    auto cap = [&](int64_t n) { return (unsigned)(up.p2m_grid > 0 ? std::min<int64_t>(n, up.p2m_grid) : n); };
    constexpr size_t s1 = sizeof(P2MShared<real, P, true>), s0 = sizeof(P2MShared<real, P, false>);
    constexpr size_t sc = sizeof(ClimbShared<real, P>);
    if constexpr (s0 > 40 * 1024 || sc > 40 * 1024) {
        PGB_CUDA(cudaFuncSetAttribute(k_p2m<real, P, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s1));
        PGB_CUDA(cudaFuncSetAttribute(k_p2m<real, P, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s0));
        PGB_CUDA(cudaFuncSetAttribute(k_climb<real, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sc));
    }
    if (up.pmom) k_p2m<real, P, true><<<cap(up.n_leaves), p2m_threads(P), s1, s>>>(up, (real*)mom);
    else k_p2m<real, P, false><<<cap(up.n_leaves), p2m_threads(P), s0, s>>>(up, (real*)mom);
    if (up.n_internal > 0) k_climb<real, P><<<cap(up.n_internal), 256 * climb_wpc(P, sizeof(real)), sc, s>>>(up, (real*)mom);
    if (up.n_nodes <= 0) return;
    launch_far<real, P>(up, mom, s);
}

}  // namespace pgb
