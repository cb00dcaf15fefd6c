// P2P of the double-single product (PGB_FP64_DS): the far rule point by point.
//
// The FP32 and FP64 kernels sum panel by panel (treecode.cuh, panel_sums).  In
// double-single that form rounds |d|^2 and n.d once for all points of a panel,
// and seven points with one common error no longer average it: products lay
// 2.7e-15 to 4.9e-15 (relative, 2-norm) from the FP64 ones.  So here every
// point has its own position, squared distance and normal product, and the
// target's offset from a leaf's centre is formed in FP64 and split once a leaf:
// 1.1e-15 to 3.0e-15 over the same six systems (one unit of a pair is 3.6e-15).
// Kept from the leaf's centre because the points' rounding is then of the leaf's
// size; from the group's centre 1.5e-15 to 3.4e-15, with offsets added as pairs
// 2.2e-15 to 3.9e-15.
#pragma once
#include "treecode.cuh"

namespace pgb {

// One point {y, q_L}, {p n, q_Y} for one target at x, both relative to the
// leaf's centre: U_L += q_L / r - p n.(x - y) / r^3 and the Yukawa counterpart.
// Differences, the normal product, the exponent's argument and the sums are
// renormalised; the products between them need not be (1.91 -> 1.81 ms for the
// product below and the same distances from FP64 to 5 %; with none renormalised
// 1.3e-15 to 3.1e-15).
template <bool LAP>
__device__ __forceinline__ void ds_point(const ds4& A, const ds4& B, bool own, ds x, ds y, ds z, ds kappa, ds nkl,
                                         ds& UL, ds& UY) {
    const ds dx = x - A.x, dy = y - A.y, dz = z - A.z;
    const ds r2 = ds_fma(dx, dx, ds_fma_u(dy, dy, ds_mul_u(dz, dz)));
    ds ri = ds_rsqrt(r2);
    if (own) ri = ds(0);  // the panel's own integral is a near-field correction
    const ds t = ds_mul_u(ds_fma(B.x, dx, ds_fma(B.y, dy, B.z * dz)), ds_mul_u(ri, ri));
    const ds r = ds_mul_u(r2, ri);
    const ds e = ds_mul_u(ds_exp2(nkl * r), ri);
    if (LAP) UL = ds_fma(ri, ds_add_u(A.w, -t), UL);
    UY = ds_fma(e, ds_fma_u(-ds_fma_u(kappa, r, ds(1)), t, B.w), UY);
}

// Points summed plainly before they join an item's sums: their additions round
// at the size of a run's sum (one run of 32: a few per cent more error).
#define P2P_DS_RUN 16

// Work items, columns and warps as k_p2p; a warp stages 32 points at a time,
// one per lane.  Bound by FP32 operations, about 230 a point with the Laplace
// kernel: product of 36200 panels 1.81 ms (panel by panel 1.51; before it, with
// slower functions, 2.55; two points at a time 1.96 -> 1.91 then).
template <int K, int NW>
__global__ void __launch_bounds__(NW * 32) k_p2p_ds(EvalArgs a, const dbl4* __restrict__ xrel) {
    __shared__ __align__(16) ds4 sA[NW][32], sB[NW][32];
    __shared__ int sJ[NW][32], sN[NW][32];  // panel, leaf node
    __shared__ ds red[NW][4][32];
    __shared__ int64_t s_item;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned long long dm = body_mask(a.bmask), act = a.src_mask & dm;
    const ds kappa = ds_from_double(a.kappa);
    const ds nkl = exp_scale(kappa);
    const dbl4* __restrict__ pd = (const dbl4*)a.pd;
    const double* __restrict__ pg = (const double*)a.pg;
    for (int64_t it = next_item(a.p2p_work, -1, &s_item); it < a.n_pitems; it = next_item(a.p2p_work, it, &s_item)) {
        const int64_t g = a.pitem_group[it];
        const int gb = a.gbody[g];
        if (!(((a.tgt_mask & dm) >> gb) & 1ull) || g < a.g_lo || g >= a.g_hi) continue;  // rows not used (block-uniform)
        const int p0 = a.gstart[g], p1 = a.gend[g];
        const int p = p0 + lane;
        const dbl4 xr = xrel[p < p1 ? p : p0];
        const double gc0 = a.gcenter[3 * g], gc1 = a.gcenter[3 * g + 1], gc2 = a.gcenter[3 * g + 2];
        const bool glap = a.lap_body[gb];
        ds UL = ds(0), UY = ds(0);
        ds x = ds(0), y = ds(0), z = ds(0);  // the target relative to the centre of leaf `leaf`
        int leaf = -1;
        const int64_t i0 = a.pitem_off[g], c0 = a.col_off[g], nc = a.col_off[g + 1] - c0;
        const int64_t per = (nc + a.pitem_off[g + 1] - i0 - 1) / (a.pitem_off[g + 1] - i0);
        const int64_t b0 = c0 + (it - i0) * per, b1 = min(c0 + nc, b0 + per);
        const int64_t wper = b1 > b0 ? (b1 - b0 + NW - 1) / NW : 0;
        const int64_t w0 = b0 + w * wper;
        const int np = K * (int)max((int64_t)0, min(b1, w0 + wper) - w0);
        for (int e = 0; e < np; e += 32) {
            const int cnt = min(32, np - e);
            bool lap = false, on = false;
            const int c = (e + lane) / K, m = e + lane - c * K;
            int j = -1, b = 0;
            if (lane < cnt) {
                j = __float_as_int(column(a, g, c0, w0 - c0 + c).w);
                b = a.pbody[j];
                on = (act >> b) & 1ull;
            }
            if (!__any_sync(0xffffffffu, on)) continue;  // (as k_p2p)
            __syncwarp();
            if (lane < cnt) {
                lap = glap && b == gb;
                const double wt = on ? a.rule.w[K == 3 ? 1 : (m + 2) / 3] : 0.0;
                const dbl4 d = pd[j], v = a.pts[(int64_t)j * K + m];
                const double* n = pg + 16 * (int64_t)j + 12;
                const double ph = wt * d.z;
                sA[w][lane] = cvt4<ds>(dbl4{v.x, v.y, v.z, wt * d.x});
                sB[w][lane] = cvt4<ds>(dbl4{ph * n[0], ph * n[1], ph * n[2], wt * d.y});
                sJ[w][lane] = j;
                sN[w][lane] = a.pnode[j];
            }
            const unsigned laps = __ballot_sync(0xffffffffu, lap);
            __syncwarp();
#pragma unroll 1
            for (int k0 = 0; k0 < cnt; k0 += P2P_DS_RUN) {
                ds sL = ds(0), sY = ds(0);
                const int k1 = min(cnt, k0 + P2P_DS_RUN);
#pragma unroll 2
                for (int k = k0; k < k1; ++k) {
                    if (sN[w][k] != leaf) {
                        leaf = sN[w][k];
                        x = ds_from_double(xr.x - (a.ncenter[3 * leaf] - gc0));
                        y = ds_from_double(xr.y - (a.ncenter[3 * leaf + 1] - gc1));
                        z = ds_from_double(xr.z - (a.ncenter[3 * leaf + 2] - gc2));
                    }
                    const bool own = sJ[w][k] == p;
                    if ((laps >> k) & 1u) ds_point<true>(sA[w][k], sB[w][k], own, x, y, z, kappa, nkl, sL, sY);
                    else ds_point<false>(sA[w][k], sB[w][k], own, x, y, z, kappa, nkl, sL, sY);
                }
                if (laps) UL = UL + sL;
                UY = UY + sY;
            }
        }
        store_item<ds, NW>(red, w, lane, UL, ds(0), UY, ds(0), a.Up + 64 * it);
    }
}

inline void launch_p2p_ds(const EvalArgs& ev, int K, const void* xrel, cudaStream_t s) {
    constexpr int NW = 8;
    if (ev.n_pitems <= 0) return;
    const unsigned grid = (unsigned)(ev.p2p_work ? ev.persist_blocks : ev.n_pitems);
    const dbl4* x = (const dbl4*)xrel;
    switch (K) {
        case 1: k_p2p_ds<1, NW><<<grid, NW * 32, 0, s>>>(ev, x); break;
        case 3: k_p2p_ds<3, NW><<<grid, NW * 32, 0, s>>>(ev, x); break;
        case 4: k_p2p_ds<4, NW><<<grid, NW * 32, 0, s>>>(ev, x); break;
        case 7: k_p2p_ds<7, NW><<<grid, NW * 32, 0, s>>>(ev, x); break;
        default: fail(PGB_EINVAL, "K must be 1, 3, 4 or 7");
    }
}

}  // namespace pgb
