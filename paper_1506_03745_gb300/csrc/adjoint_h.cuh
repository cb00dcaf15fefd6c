// Transposed treecode in FP64 (the adjoint operator A^T, see adjoint.cuh) in the
// harmonic basis of the far field: the forward product sums B_j(x_i - c_b)
// sum_k tab_jk M_k(b) (farfield.cu), so its transpose gathers per node
//   H_j(b) = sum over the pairs (g, b) of sum_{i in g} s_i B_j(x_i - c_b)
// (k_m2p_TH), forms L_k(b) = sum_j tab_jk H_j(b) (k_far_TH), pushes L down the
// tree by the binomial shift (k_l2l_TH) and meets the panel moments
// V_k = sum_m w_m u_m^k of the leaves' panels: sum_s w_s Phi(y_s) = A sum_k L_k V_k
// and sum_s w_s n . grad_y Phi = -A sum_k V_k sum_a n_a (k_a + 1) L_{k + e_a}
// (k_l2p_TH).  Within a solve the near field is the stored one, read the other
// way (k_near_T).  5380 panels, one product: gather 1.89 ms with Taylor
// coefficients, 0.42 in the harmonic basis with both kernels' sums sharing the
// recurrences (0.48 one after the other), near field 3.88 ms formed anew, 0.06
// read, nodes 0.26 ms; the whole
// gradient 606 -> 74 ms.  (The FP32 product keeps the kernels of adjoint.cuh,
// whose sums, up to the order of their atomic additions, an FP32 gradient's
// derivatives rest on.)
#pragma once
#include "adjoint.cuh"

namespace pgb {

// The harmonic basis values of one pair, s B_j for j = 0 .. n_far(P) - 1 in the
// order of far_pos, handed to putY / putL (std::integral_constant j, value):
// Yukawa sY e^{-x} / r h_l q_{l,m} (Re, Im) and, with LAP, Laplace
// sL / r r^{-l} q_{l,m} (Re, Im), which share the recurrences of q.
template <typename real, int P, bool LAP, class FY, class FL>
__device__ __forceinline__ void far_basis(real Rx, real Ry, real Rz, real kappa, real sY, real sL, FY&& putY, FL&& putL) {
    const real r2 = Rx * Rx + Ry * Ry + Rz * Rz;
    const real ri = rsqrt_(r2);
    const real nx = Rx * ri, ny = Ry * ri, nz = Rz * ri;
    real h[P + 1], g[P + 1];
    h[0] = exp_(-kappa * (r2 * ri)) * ri * sY;
    g[0] = ri * sL;
    if constexpr (P >= 1) {
        h[1] = -(ri + kappa) * h[0];
        g[1] = ri * g[0];
    }
    static_for<2, P + 1>([&](auto Lc) {
        constexpr int l = decltype(Lc)::value;
        h[l] = (kappa * kappa) * h[l - 2] - (real(2 * l - 1) * ri) * h[l - 1];
        if constexpr (LAP) g[l] = ri * g[l - 1];
    });
    real X = real(1), Y = real(0);
    static_for<0, P + 1>([&](auto M) {
        constexpr int m = decltype(M)::value;
        real q0 = real(1), q1 = real(0);
        static_for<m, P + 1>([&](auto Lc) {
            constexpr int l = decltype(Lc)::value;
            if constexpr (l > m) {
                const real q = l == m + 1 ? nz : nz * q0 - real(far_c(l - 1, m)) * q1;
                q1 = q0;
                q0 = q;
            }
            const real w = l > m ? h[l] * q0 : h[l];
            const real v = !LAP ? real(0) : l > m ? g[l] * q0 : g[l];
            constexpr std::integral_constant<int, far_pos(P, l, m, 0)> j0{};
            if constexpr (m == 0) {
                putY(j0, w);
                if constexpr (LAP) putL(j0, v);
            } else {
                constexpr std::integral_constant<int, far_pos(P, l, m, 1)> j1{};
                putY(j0, w * X);
                putY(j1, w * Y);
                if constexpr (LAP) {
                    putL(j0, v * X);
                    putL(j1, v * Y);
                }
            }
        });
        if constexpr (m == 0) {
            X = nx;
            Y = ny;
        } else {
            const real xn = nx * X - ny * Y;
            Y = nx * Y + ny * X;
            X = xn;
        }
    });
}

// Sums over the warp of one pair's basis values, added to dst (atomic: the
// forward pairs (g, b) of one node b are spread over blocks); 32 at a time.
template <typename real, int P, bool LAP>
__device__ __forceinline__ void gather_basis(real Rx, real Ry, real Rz, real kappa, real sY, real sL, real* dst) {
    constexpr int NC = n_far(P), PAD = n_far_pad(P);
    const int lane = threadIdx.x & 31;
    real v[32], u[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = u[k] = real(0);
    auto put = [&](real (&b)[32], real* d, auto J, real x) {
        constexpr int j = decltype(J)::value;
        b[j & 31] = x;
        if constexpr ((j & 31) == 31 || j == NC - 1) {
            constexpr int b0 = j & ~31;
            const real sum = reduce_scatter32(b);
            if (b0 + lane <= j) atomicAdd(d + b0 + lane, sum);
        }
    };
    far_basis<real, P, LAP>(
        Rx, Ry, Rz, kappa, sY, sL, [&](auto J, real x) { put(v, dst + PAD, J, x); },
        [&](auto J, real x) { put(u, dst, J, x); });
}

// Far gather: one block of NW warps per forward M2P work item (up to m2p_item
// far nodes of one target group, as k_m2p); lane = target i with weights
// (s_L, s_Y); per node b the harmonic values of the 32 targets are summed and
// added to H(b) (n_far_pad(P) Laplace, then as many Yukawa).  In the Cartesian
// basis a pair's Taylor coefficients cost 2231 operations and 84 sums per
// kernel; here about 200 and 49, bound by FP64 operations.
template <typename real, int P, int NW>
__global__ void __launch_bounds__(NW * 32) k_m2p_TH(TArgs a, const typename V4<real>::t* __restrict__ xrel,
                                                    const double* __restrict__ sT, real* __restrict__ H) {
    using v4 = typename V4<real>::t;
    constexpr int NC = n_far_pad(P);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t it = blockIdx.x;
    if (it >= a.n_fitems) return;
    const int64_t g = a.fitem_group[it];
    const int64_t p0 = a.gstart[g], p1 = a.gend[g];
    const int64_t p = p0 + lane;
    const bool active = p < p1;
    const v4 xr = active ? xrel[p] : xrel[p0];
    const real sL = active ? (real)sT[2 * p] : real(0), sY = active ? (real)sT[2 * p + 1] : real(0);
    const double gc0 = a.gcenter[3 * g], gc1 = a.gcenter[3 * g + 1], gc2 = a.gcenter[3 * g + 2];
    const int gb = a.gbody[g];
    const real kappa = (real)a.kappa;
    const int64_t fb = a.far_off[g] + (it - a.fitem_off[g]) * a.m2p_item;
    const int64_t f1 = min(a.far_off[g + 1], fb + a.m2p_item);
    for (int64_t e = fb + w; e < f1; e += NW) {
        const int nd = a.far_l[e];
        const real Rx = xr.x - (real)(a.ncenter[3 * nd] - gc0), Ry = xr.y - (real)(a.ncenter[3 * nd + 1] - gc1),
                   Rz = xr.z - (real)(a.ncenter[3 * nd + 2] - gc2);
        real* h = H + (int64_t)nd * 2 * NC;
        if ((a.nbody[nd] == gb) && a.lap_body[gb]) gather_basis<real, P, true>(Rx, Ry, Rz, kappa, sY, sL, h);
        else gather_basis<real, P, false>(Rx, Ry, Rz, kappa, sY, sL, h);
    }
}

// L_k = sum_j tab_jk H_j for every node (T Laplace then T Yukawa, as the
// moments): one block per node, a thread per k and kernel.
template <typename real, int P>
__global__ void __launch_bounds__(128) k_far_TH(TArgs a, int64_t n_nodes, const real* __restrict__ H,
                                               real* __restrict__ Lmom) {
    constexpr int T = MI<P>::T, TR = far_cols(P), NC = n_far_pad(P);
    __shared__ real sh[2 * NC];
    const int64_t nd = blockIdx.x;
    for (int k = threadIdx.x; k < 2 * NC; k += blockDim.x) sh[k] = H[nd * 2 * NC + k];
    __syncthreads();
    const real* __restrict__ tab = (const real*)a.far_tr;
    for (int q = threadIdx.x; q < 2 * T; q += blockDim.x) {
        const bool yuk = q >= T;
        const int k = yuk ? q - T : q;
        const real* h = sh + (yuk ? NC : 0);
        const real* col = tab + (yuk ? 0 : (size_t)TR * T) + k;
        real s = 0;
        int l = 0, r = 0;  // column j = l^2 + r
#pragma unroll 8
        for (int j = 0; j < n_far(P); ++j) {
            const int m = (r + 1) / 2;
            s += col[(size_t)j * T] * h[far_pos(P, l, m, r ? (r - 1) & 1 : 0)];
            if (++r > 2 * l) {
                r = 0;
                ++l;
            }
        }
        Lmom[nd * 2 * T + q] = s;
    }
}

// Downward shift into the nodes of one level: L_j(child) +=
// sum_{k >= j} C(k, j) (c - c_child)^{k - j} L_k(c), one warp per child, along
// each axis the lines of up_m2m with the transposed recurrence
// s_k += d s_{k+1}, k = t..n-1, for t = n-1..0 in registers (Taylor shift).
template <typename real, int P>
__global__ void __launch_bounds__(128) k_l2l_TH(TArgs a, const int32_t* __restrict__ parent,
                                                   real* __restrict__ Lmom) {
    constexpr int T = MI<P>::T, NL = (P + 1) * (P + 2) / 2;
    __shared__ real buf[4][2 * T];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t ch = a.lvl_begin + (int64_t)blockIdx.x * 4 + w;
    if (ch >= a.lvl_end) return;  // warp-uniform
    const int par = parent[ch];
    if (par < 0) return;
    real* b = buf[w];
    for (int k = lane; k < 2 * T; k += 32) b[k] = Lmom[(int64_t)par * 2 * T + k];
    real d3[3];
    for (int c = 0; c < 3; ++c) d3[c] = (real)(a.ncenter[3 * par + c] - a.ncenter[3 * ch + c]);
    __syncwarp();
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const Pair<real> d{d3[ax], d3[ax]};
#pragma unroll 1
        for (int i = lane; i < NL; i += 32) {
            int s0 = 0, r = i;  // (e, f) by e + f = 0..P, the longest lines first
            while (r > s0) r -= ++s0;
            const int e = r, f = s0 - r, n = P - s0;
            Pair<real> s[P + 1];
            int at[P + 1];
#pragma unroll
            for (int k = 0; k <= P; ++k) {
                at[k] = ax == 0 ? mi_index(k, e, f) : (ax == 1 ? mi_index(e, k, f) : mi_index(e, f, k));
                s[k] = k <= n ? Pair<real>{b[at[k]], b[T + at[k]]} : Pair<real>{real(0), real(0)};
            }
#pragma unroll
            for (int t = 0; t < P; ++t)
#pragma unroll
                for (int k = P - 1; k >= t; --k) s[k] = pair_fma(d, s[k + 1], s[k]);
#pragma unroll
            for (int k = 0; k <= P; ++k)
                if (k <= n) {
                    b[at[k]] = s[k].a;
                    b[T + at[k]] = s[k].b;
                }
        }
        __syncwarp();
    }
    for (int k = lane; k < 2 * T; k += 32) Lmom[ch * 2 * T + k] += b[k];
}

// Far field at the panels of every leaf (one block per leaf, a warp per panel
// in turn): the columns' sums over the panel's points / area (see above) from
// the panel moments, into pan (V_L, K_L, V_Y, K_Y).
template <typename real, int P, bool STORED>
__global__ void __launch_bounds__(128) k_l2p_TH(TArgs a, UpArgs u, const real* __restrict__ Lmom) {
    constexpr int T = MI<P>::T;
    __shared__ real sL[2][4][T];  // per kernel: L_k, then (k_a + 1) L_{k + e_a}
    __shared__ real pw[STORED ? 1 : UP_FLY * 7][3][P + 1];  // powers at the points of four panels
    const int nd = a.leaf_node[blockIdx.x];
    for (int q = threadIdx.x; q < 2 * T; q += blockDim.x) {
        const int t = q >= T, k = t ? q - T : q;
        const real* L = Lmom + (int64_t)nd * 2 * T + (t ? T : 0);
        int x, y, z;
        decode_mi(k, x, y, z);
        const bool in = x + y + z < P;
        sL[t][0][k] = L[k];
        sL[t][1][k] = in ? real(x + 1) * L[mi_index(x + 1, y, z)] : real(0);
        sL[t][2][k] = in ? real(y + 1) * L[mi_index(x, y + 1, z)] : real(0);
        sL[t][3][k] = in ? real(z + 1) * L[mi_index(x, y, z + 1)] : real(0);
    }
    __syncthreads();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const real* __restrict__ pg = (const real*)u.pg;
    const real* __restrict__ pm = (const real*)u.pmom;
    for (int64_t jb = a.nstart[nd]; jb < a.nend[nd]; jb += 4) {
        const int64_t j = jb + w;
        if constexpr (!STORED) {
            __syncthreads();
            stage_powers<real, P>(u, jb, (int)min((int64_t)4, a.nend[nd] - jb), pw);
            __syncthreads();
        }
        if (j >= a.nend[nd]) continue;
        const real n0 = pg[16 * j + 12], n1 = pg[16 * j + 13], n2 = pg[16 * j + 14];
        real v[4] = {0, 0, 0, 0};
        for (int k = lane; k < T; k += 32) {
            real m;
            if constexpr (STORED) {
                m = pm[j * T + k];
            } else {
                int x, y, z;
                decode_mi(k, x, y, z);
                m = panel_moment<real, P>(u, pw + w * u.K, x, y, z);
            }
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                v[2 * t] += m * sL[t][0][k];
                v[2 * t + 1] += m * (n0 * sL[t][1][k] + n1 * sL[t][2][k] + n2 * sL[t][3][k]);
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = warp_sum(v[c]);
        if (lane < 4) {
            const real x = lane == 0 ? v[0] : lane == 1 ? -v[1] : lane == 2 ? v[2] : -v[3];
            a.pan[4 * j + lane] = (double)x;
        }
    }
}

// Near field, transposed, from the stored matrix: one block per source leaf;
// its warps take the forward near entries (g, leaf) in turn, lane = target of
// g, eight of the leaf's panels at a time, and the sums over targets and warps
// follow at the end (fixed order).  nearp: V_L, K_L, V_Y, K_Y columns / area.
template <int NW>
__global__ void __launch_bounds__(NW * 32) k_near_T(TArgs a, const double* __restrict__ sT) {
    constexpr int PC = 8;
    __shared__ double red[NW][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nd = a.leaf_node[blockIdx.x];
    const int nb = a.nbody[nd];
    const int j0 = a.nstart[nd], np = a.nend[nd] - j0;
    const int64_t t0 = a.tn_off[nd], t1 = a.tn_off[nd + 1];
    const NearGroup* __restrict__ ng = (const NearGroup*)a.near_grp;
    const double* __restrict__ mat = (const double*)a.near_mat;
    for (int c0 = 0; c0 < np; c0 += PC) {
        const int n = min(PC, np - c0);
        double acc[32];  // panel q, column c at 4 q + c
#pragma unroll
        for (int q = 0; q < 32; ++q) acc[q] = 0;
        for (int64_t t = t0 + w; t < t1; t += NW) {
            const int64_t e = a.tn_e[t];
            const int g = a.near_group[e];
            const int p = a.gstart[g] + lane;
            const bool on = p < a.gend[g];
            const double2 s2 = on ? reinterpret_cast<const double2*>(sT)[p] : make_double2(0.0, 0.0);
            const double sL = s2.x, sY = s2.y;
            const NearGroup nm = ng[g];
            const int64_t c = a.ent_col[e] + c0;
            const double* u = mat + 64 * near_unit(nm, c);
            if (nb == a.gbody[g] && a.lap_body[nb]) {
#pragma unroll
                for (int q = 0; q < PC; ++q) {
                    const double* x = u + 128 * (int64_t)min(q, n - 1);
                    const double2 m = reinterpret_cast<const double2*>(x)[lane];
                    const double2 o = reinterpret_cast<const double2*>(x)[32 + lane];
                    acc[4 * q] += sL * m.x;
                    acc[4 * q + 1] += sL * m.y;
                    acc[4 * q + 2] += sY * o.x;
                    acc[4 * q + 3] += sY * o.y;
                }
            } else {
#pragma unroll
                for (int q = 0; q < PC; ++q) {
                    const double* x = u + 64 * (int64_t)min(q, n - 1) + 2 * lane;
                    acc[4 * q + 2] += sY * x[0];
                    acc[4 * q + 3] += sY * x[1];
                }
            }
        }
        red[w][lane] = reduce_scatter32(acc);
        __syncthreads();
        if (w == 0 && lane < 4 * n) {
            double s = 0;
            for (int k = 0; k < NW; ++k) s += red[k][lane];
            a.nearp[4 * (int64_t)(j0 + c0) + lane] = s;
        }
        __syncthreads();
    }
}

}  // namespace pgb
