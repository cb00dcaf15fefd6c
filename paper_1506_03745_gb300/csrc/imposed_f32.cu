// The imposed-boundary terms of an FP32 gradient, b_known of one surface with
// its imposed value set to one (pgb_grad: dF/dsigma0 and dF/dphi0 take
// lam . b_known).  They are one FP32 product per surface and gradient, and the
// derivative carries that product's rounding, 1e-9 to 4e-9 of its value against
// the double-single product's.  The sums here are formed point by point, with
// Cartesian moments and monomials, in one fixed order; the products of the
// solve, in another order, or the double-single one move the derivative by that
// much, ten times and more what two runs of one gradient differ in it (1e-11 to
// 6e-10, from the atomic additions of the adjoint solve).  So that an FP32
// gradient's derivative in an imposed value stays what it was, this path keeps
// its arithmetic; it is 0.3 ms of a gradient of 36000 panels.  Orders 0..8 (as
// pgb_grad), Yukawa kernel only: imposed densities live on surfaces, and the
// Laplace kernel couples a molecule only to itself.
#include <algorithm>

#include "treecode.cuh"

namespace pgb {

static inline int nblk(int64_t n, int t) { return (int)std::max<int64_t>(1, (n + t - 1) / t); }

namespace {

struct ImpArgs {
    int body;                      // the surface
    int K;
    double kappa;
    int64_t n_groups;
    const int32_t *gstart, *gend;
    const int32_t *nstart, *nend, *nbody, *nchild, *child, *leaf_node;
    const double* ncenter;
    const float4* src;             // per point {y - leaf centre, unused}, {w phi n, w psi_Y}
    const float* tab;              // far-field table, transposed: tab[k TR + j]
    float *mom, *far;              // T moments, n_pad coefficients per node
};

// Densities of the surface (psi_Y, phi per panel, zero elsewhere) and its point
// source terms.
__global__ void k_imp_src(Geo g, BodyDev bd, int body, double eps_out, const float4* __restrict__ yrel,
                          float4* __restrict__ src, float2* __restrict__ dens) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= g.n_pan) return;
    const int b = g.pbody[i];
    double psiY = 0, phi = 0;
    if (b == body) {
        if (bd.kind[b] == PGB_SET_POTENTIAL) phi = bd.bc[b];
        else if (bd.kind[b] == PGB_SET_CHARGE) psiY = -bd.bc[b] / eps_out;
    }
    const float rY = (float)psiY, rp = (float)phi;
    dens[i] = make_float2(rY, rp);
    const float nx = (float)g.n[3 * i], ny = (float)g.n[3 * i + 1], nz = (float)g.n[3 * i + 2];
    for (int m = 0; m < g.K; ++m) {
        const int64_t p = i * g.K + m;
        const float w = (float)g.w[p];
        float4 A = yrel[p], B;
        const float wp = w * rp;
        A.w = 0.f;
        B.x = wp * nx;
        B.y = wp * ny;
        B.z = wp * nz;
        B.w = w * rY;
        src[2 * p] = A;
        src[2 * p + 1] = B;
    }
}

// P2M of the surface's leaves: a thread per multi-index.
template <int P>
__global__ void __launch_bounds__(256) k_imp_p2m(ImpArgs a) {
    constexpr int T = MI<P>::T;
    __shared__ float pw[128][3][P + 1], sq[128][4], sd[3][T];
    const int nd = a.leaf_node[blockIdx.x];
    if (a.nbody[nd] != a.body) return;
    const int tid = threadIdx.x;
    int x = 0, y = 0, z = 0;
    const bool on = tid < T;
    if (on) decode_mi(tid, x, y, z);
    const bool low = on && x + y + z < P;
    float qY = 0, dx = 0, dy = 0, dz = 0;
    const int64_t s0 = (int64_t)a.nstart[nd] * a.K, s1 = (int64_t)a.nend[nd] * a.K;
    for (int64_t t = s0; t < s1; t += 128) {
        const int cnt = (int)min((int64_t)128, s1 - t);
        __syncthreads();
        if (tid < cnt) {
            const float4 A = a.src[2 * (t + tid)], B = a.src[2 * (t + tid) + 1];
            const float u[3] = {-A.x, -A.y, -A.z};
            for (int q = 0; q < 3; ++q) {
                float v = 1;
                for (int m = 0; m <= P; ++m) {
                    pw[tid][q][m] = v;
                    v = v * u[q];
                }
            }
            sq[tid][0] = B.w;
            sq[tid][1] = B.x;
            sq[tid][2] = B.y;
            sq[tid][3] = B.z;
        }
        __syncthreads();
        if (on)
            for (int j = 0; j < cnt; ++j) {
                const float mono = pw[j][0][x] * pw[j][1][y] * pw[j][2][z];
                qY += sq[j][0] * mono;
                if (low) {
                    dx += sq[j][1] * mono;
                    dy += sq[j][2] * mono;
                    dz += sq[j][3] * mono;
                }
            }
    }
    __syncthreads();
    if (on) {
        sd[0][tid] = dx;
        sd[1][tid] = dy;
        sd[2][tid] = dz;
    }
    __syncthreads();
    if (!on) return;
    float dl = 0;
    if (x) dl += float(x) * sd[0][mi_index(x - 1, y, z)];
    if (y) dl += float(y) * sd[1][mi_index(x, y - 1, z)];
    if (z) dl += float(z) * sd[2][mi_index(x, y, z - 1)];
    a.mom[(int64_t)nd * T + tid] = qY + dl;
}

// Moment shift into the nodes [lo, hi) of one level, three one-axis passes, the
// children summed in order.
template <int P>
__global__ void __launch_bounds__(256) k_imp_m2m(ImpArgs a, int64_t lo) {
    constexpr int T = MI<P>::T;
    __shared__ float buf[2][T], cd[3][P + 1];
    const int64_t nd = lo + blockIdx.x;
    const int nc = a.nchild[nd], fc = a.child[nd];
    if (nc == 0 || a.nbody[nd] != a.body) return;
    const int tid = threadIdx.x;
    int kx[3] = {0, 0, 0};
    if (tid < T) decode_mi(tid, kx[0], kx[1], kx[2]);
    float acc = 0.f;
    for (int c = 0; c < nc; ++c) {
        __syncthreads();
        if (tid < T) buf[0][tid] = a.mom[(int64_t)(fc + c) * T + tid];
        if (tid < 3) {
            const float d = (float)(a.ncenter[3 * nd + tid] - a.ncenter[3 * (fc + c) + tid]);
            float v = 1;
            for (int m = 0; m <= P; ++m) {
                cd[tid][m] = v;
                v = v * d;
            }
        }
        __syncthreads();
        for (int ax = 0; ax < 3; ++ax) {
            const float* s = buf[ax & 1];
            float* d = buf[(ax + 1) & 1];
            if (tid < T) {
                float sum = 0;
                int binom = 1;  // C(ka, j)
                for (int j = 0; j <= kx[ax]; ++j) {
                    const int jx = ax == 0 ? j : kx[0], jy = ax == 1 ? j : kx[1], jz = ax == 2 ? j : kx[2];
                    const float coef = (float)binom * cd[ax][kx[ax] - j];
                    sum += coef * s[mi_index(jx, jy, jz)];
                    binom = binom * (kx[ax] - j) / (j + 1);
                }
                d[tid] = sum;
            }
            __syncthreads();
        }
        if (tid < T) acc += buf[1][tid];
    }
    if (tid < T) a.mom[nd * T + tid] = acc;
}

// Monomial far-field coefficients (the table of pgb_far_table) of every node.
template <int P>
__global__ void __launch_bounds__(256) k_imp_far(ImpArgs a) {
    constexpr int T = MI<P>::T, TP = n_mono_pad(P), TR = mono_cols(P);
    __shared__ float m[T];
    const int64_t nd = blockIdx.x;
    if (a.nbody[nd] != a.body) return;
    for (int k = threadIdx.x; k < T; k += blockDim.x) m[k] = a.mom[nd * T + k];
    __syncthreads();
    const int j = threadIdx.x;
    const float* __restrict__ tab = a.tab + j;
    float acc0 = 0.f, acc1 = 0.f;
#pragma unroll 8
    for (int k = 0; k + 1 < T; k += 2) {
        acc0 += m[k] * __ldg(tab + (size_t)k * TR);
        acc1 += m[k + 1] * __ldg(tab + (size_t)(k + 1) * TR);
    }
    if (T & 1) acc0 += m[T - 1] * __ldg(tab + (size_t)(T - 1) * TR);
    if (j < TP) a.far[nd * TP + j] = acc0 + acc1;
}

// index of S^(a,b,0) in the evaluation order of order P
__host__ __device__ constexpr int eval_index(int P, int a, int b) {
    int o = 0;
    for (int q = 0; q < a; ++q) o += (P - q + 1) * (P - q + 2) / 2;
    for (int q = 0; q < b; ++q) o += P - a - q + 1;
    return o;
}
template <int P>
__device__ __forceinline__ float imp_eval(float Rx, float Ry, float Rz, float kappa, const float* __restrict__ cY) {
    const float r2 = Rx * Rx + Ry * Ry + Rz * Rz;
    const float ri = rsqrt_(r2);
    const float i2 = ri * ri;
    const float sx = Rx * i2, sy = Ry * i2, sz = Rz * i2;
    float acc[P + 1];
#pragma unroll
    for (int p = 0; p <= P; ++p) acc[p] = 0.f;
    float xa = 1.f;
    static_for<0, P + 1>([&](auto A) {
        constexpr int a = decltype(A)::value;
        float xy = xa;
        static_for<0, P - a + 1>([&](auto Bc) {
            constexpr int b = decltype(Bc)::value;
            constexpr int i0 = eval_index(P, a, b);
            float t = xy;
            static_for<0, P - a - b + 1>([&](auto Cc) {
                constexpr int c = decltype(Cc)::value;
                acc[a + b + c] = acc[a + b + c] + cY[i0 + c] * t;
                if constexpr (c < P - a - b) t = t * sz;
            });
            if constexpr (b < P - a) xy = xy * sy;
        });
        if constexpr (a < P) xa = xa * sx;
    });
    const float r = r2 * ri;
    const float x = kappa * r;
    const float x2 = x * x;
    float u = acc[0];
    float gm2 = 1.f, gm1 = -(x + 1.f);
    if (P >= 1) u = u + gm1 * acc[P >= 1 ? 1 : 0];
#pragma unroll
    for (int p = 2; p <= P; ++p) {
        const float g = -(float(2 * p - 1) * gm1) + x2 * gm2;
        u = u + g * acc[p];
        gm2 = gm1;
        gm1 = g;
    }
    return (exp_(-x) * ri) * u;
}

// Block sum of the warps' compensated pairs, in warp order, per lane.
__device__ __forceinline__ void imp_store(float (*red)[2][32], int w, int lane, float U, float c, double* out) {
    red[w][0][lane] = U;
    red[w][1][lane] = c;
    __syncthreads();
    if (w == 0) {
        float s = 0, e = 0;
        for (int k = 0; k < 8; ++k) {
            kadd(s, e, red[k][0][lane]);
            kadd(s, e, red[k][1][lane]);
        }
        out[lane] = (double)s + (double)e;
    }
}

// P2P tiles of a group: its near leaves in runs of 32 points.
__global__ void k_imp_tile_count(ImpArgs a, const int64_t* noff, const int32_t* nearl, int64_t* cnt) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= a.n_groups) return;
    int64_t c = 0;
    for (int64_t e = noff[g]; e < noff[g + 1]; ++e)
        c += ((int64_t)(a.nend[nearl[e]] - a.nstart[nearl[e]]) * a.K + 31) / 32;
    cnt[g] = c;
}
__global__ void k_imp_tile_fill(ImpArgs a, const int64_t* noff, const int32_t* nearl, const float4* near4,
                                const int64_t* toff, float4* td, int4* tm) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= a.n_groups) return;
    int64_t t = toff[g];
    for (int64_t e = noff[g]; e < noff[g + 1]; ++e) {
        const int nd = nearl[e];
        const float4 o = near4[e];
        const int own = a.nstart[nd] < a.gend[g] && a.nend[nd] > a.gstart[g];
        const int64_t s1 = (int64_t)a.nend[nd] * a.K;
        for (int64_t q = (int64_t)a.nstart[nd] * a.K; q < s1; q += 32, ++t) {
            td[t] = make_float4(o.x, o.y, o.z, __int_as_float((int)q));
            tm[t] = make_int4(nd, (int)min((int64_t)32, s1 - q), own, a.nbody[nd]);
        }
    }
}

template <bool OWN>
__device__ __forceinline__ void imp_tile(const float4* sA, const float4* sB, int cnt, int64_t t, int64_t own_lo,
                                         int64_t own_hi, float r0x, float r0y, float r0z, float kappa, float& sumY) {
    const float nkl = -kappa * 1.4426950408889634f;
    float sY2 = 0;
#pragma unroll 4
    for (int j = 0; j < cnt; ++j) {
        const float4 A = sA[j], B = sB[j];
        const float dx = r0x - A.x, dy = r0y - A.y, dz = r0z - A.z;
        const float r2 = dx * dx + dy * dy + dz * dz;
        float ri = rsqrt_fast(r2);
        if (OWN) ri = (r2 > 0.f && !(t + j >= own_lo && t + j < own_hi)) ? ri : 0.f;
        const float pd = B.x * dx + B.y * dy + B.z * dz;
        const float tt = pd * (ri * ri);
        const float r = r2 * ri;
        const float ex = exp2_(nkl * r);
        const float gg = kappa * r + 1.f;
        if (j & 1) sY2 += (ex * ri) * (B.w - gg * tt);
        else sumY += (ex * ri) * (B.w - gg * tt);
    }
    sumY += sY2;
}

// Near and far sums of every group: one block of eight warps per group, which
// walks the group's runs of `item` tiles (then of `fitem` far entries) and adds
// their sums in run order.  U: 32 per group, near then far.
template <int P>
__global__ void __launch_bounds__(256) k_imp_eval(ImpArgs a, const int64_t* toff, const float4* td, const int4* tm,
                                                  int item, const int64_t* foff, const float4* far4, int fitem,
                                                  const float4* xrel, double* U) {
    constexpr int T = MI<P>::T, TP = n_mono_pad(P);
    (void)T;
    __shared__ float4 sA[8][32], sB[8][32];
    __shared__ float sM[8][TP];
    __shared__ float red[8][2][32];
    __shared__ double part[32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t g = blockIdx.x;
    const int64_t p0 = a.gstart[g], p1 = a.gend[g], p = p0 + lane;
    const float4 xr = p < p1 ? xrel[p] : xrel[p0];
    const float kappa = (float)a.kappa;
    const int64_t own_lo = p * a.K, own_hi = own_lo + a.K;
    double sum = 0;
    for (int64_t tb = toff[g]; tb < toff[g + 1]; tb += item) {
        const int64_t t1 = min(toff[g + 1], tb + item);
        float UY = 0, cY = 0;
        for (int64_t t = tb + w; t < t1; t += 8) {
            const float4 d = td[t];
            const int4 m = tm[t];
            float sumY = 0;
            if (m.w == a.body) {
                const int64_t first = (int64_t)__float_as_int(d.w);
                const float r0x = xr.x - d.x, r0y = xr.y - d.y, r0z = xr.z - d.z;
                __syncwarp();
                if (lane < m.y) {
                    sA[w][lane] = a.src[2 * (first + lane)];
                    sB[w][lane] = a.src[2 * (first + lane) + 1];
                }
                __syncwarp();
                if (m.z) imp_tile<true>(sA[w], sB[w], m.y, first, own_lo, own_hi, r0x, r0y, r0z, kappa, sumY);
                else imp_tile<false>(sA[w], sB[w], m.y, first, own_lo, own_hi, r0x, r0y, r0z, kappa, sumY);
            }
            kadd(UY, cY, sumY);
        }
        imp_store(red, w, lane, UY, cY, part);
        __syncthreads();
        if (w == 0) sum += part[lane];
        __syncthreads();
    }
    for (int64_t fb = foff[g]; fb < foff[g + 1]; fb += fitem) {
        const int64_t f1 = min(foff[g + 1], fb + fitem);
        float UY = 0, cY = 0;
        for (int64_t e = fb + w; e < f1; e += 8) {
            const float4 q = far4[e];
            const int nd = __float_as_int(q.w);
            if (a.nbody[nd] != a.body) continue;  // warp-uniform
            __syncwarp();
            for (int k = lane; k < TP; k += 32) sM[w][k] = a.far[(int64_t)nd * TP + k];
            __syncwarp();
            const float uY = imp_eval<P>(xr.x - q.x, xr.y - q.y, xr.z - q.z, kappa, sM[w]);
            kadd(UY, cY, uY);
        }
        imp_store(red, w, lane, UY, cY, part);
        __syncthreads();
        if (w == 0) sum += part[lane];
        __syncthreads();
    }
    if (w == 0) U[32 * g + lane] = sum;
}

// Rows: minus the sums with the near-field corrections and the jump.
__global__ void k_imp_rows(Geo g, BodyDev bd, int body, const int32_t* pan_group, const int32_t* gstart,
                           const double* __restrict__ U, const float2* __restrict__ dens,
                           const int64_t* __restrict__ coff, const int32_t* __restrict__ cj,
                           const float4* __restrict__ cval, const int64_t* __restrict__ xoff,
                           const int32_t* __restrict__ xj, const float4* __restrict__ xval, double* __restrict__ y) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= g.n_pan) return;
    const int gi = pan_group[i];
    double UY = U[32 * (int64_t)gi + (i - gstart[gi])] * (1.0 / PGB_FOUR_PI);
    float cY = 0, eY = 0;
    for (int64_t e = coff[i]; e < coff[i + 1]; ++e) {
        const float4 d = cval[e];
        const float2 s = dens[cj[e]];
        kadd(cY, eY, d.z * s.x - d.w * s.y);
    }
    for (int64_t e = xoff[i]; e < xoff[i + 1]; ++e) {
        const float4 d = xval[e];
        const float2 s = dens[xj[e]];
        kadd(cY, eY, d.z * s.x - d.w * s.y);
    }
    UY += (double)cY + (double)eY;
    const int b = g.pbody[i];
    const int64_t loc = g.perm[i] - bd.pan_off[b];
    const int64_t N = bd.pan_off[b + 1] - bd.pan_off[b];
    const int64_t o = bd.unk_off[b];
    if (bd.kind[b] == PGB_DIELECTRIC) y[o + N + loc] = -UY;
    else if (bd.kind[b] == PGB_SET_CHARGE) y[o + loc] = -UY;
    else y[o + loc] = -(UY + (b == body ? 0.5 * bd.bc[b] : 0.0));
}

template <int P>
void run(pgb_ctx* c, int body, double* y) {
    constexpr int T = MI<P>::T, TP = n_mono_pad(P), TR = mono_cols(P);
    cudaStream_t s = c->stream;
    const int64_t n = c->n_pan, ng = c->n_groups, nn = c->n_nodes;
    const Geo g = geo(c);
    const BodyDev bd = body_dev(c);
    DBuf<float4> src, td;
    DBuf<float2> dens;
    DBuf<float> mom, far;
    DBuf<int64_t> tc, toff;
    DBuf<int4> tm;
    DBuf<double> U;
    src.resize(2 * n * c->p.K);
    dens.resize(n);
    mom.resize(nn * T);
    far.resize(nn * TP);
    ImpArgs a;
    a.body = body;
    a.K = c->p.K;
    a.kappa = c->kappa;
    a.n_groups = ng;
    a.gstart = c->d_group_start;
    a.gend = c->d_group_end;
    a.nstart = c->d_node_start;
    a.nend = c->d_node_end;
    a.nbody = c->d_node_body;
    a.nchild = c->d_node_nchild;
    a.child = c->d_node_child;
    a.leaf_node = c->d_leaf_node;
    a.ncenter = c->d_node_center;
    a.src = src;
    a.tab = far_monomials_f32(c, c->kappa);
    a.mom = mom;
    a.far = far;
    k_imp_src<<<nblk(n, 128), 128, 0, s>>>(g, bd, body, c->eps_out, c->d_y32, src, dens);
    k_imp_p2m<P><<<(unsigned)c->n_leaves, 256, 0, s>>>(a);
    int launches = 5;
    for (size_t l = c->level_begin.size() - 1; l-- > 0;) {
        k_imp_m2m<P><<<(unsigned)(c->level_begin[l + 1] - c->level_begin[l]), 256, 0, s>>>(a, c->level_begin[l]);
        ++launches;
    }
    k_imp_far<P><<<(unsigned)nn, TR, 0, s>>>(a);
    tc.resize(ng);
    toff.resize(ng + 1);
    k_imp_tile_count<<<nblk(ng, 64), 64, 0, s>>>(a, c->d_near_off, c->d_near, tc);
    int64_t nt = 0;
    exclusive_scan_i64(tc, toff, ng, s, &nt);
    PGB_CUDA(cudaMemcpyAsync(toff.p + ng, &nt, 8, cudaMemcpyHostToDevice, s));
    td.resize(nt);
    tm.resize(nt);
    U.resize(32 * ng);
    k_imp_tile_fill<<<nblk(ng, 64), 64, 0, s>>>(a, c->d_near_off, c->d_near, c->d_near4, toff, td, tm);
    k_imp_eval<P><<<(unsigned)ng, 256, 0, s>>>(a, toff, td, tm, c->p.p2p_item, c->d_far_off, c->d_far4, c->p.m2p_item,
                                               c->d_x32, U);
    k_imp_rows<<<nblk(n, 128), 128, 0, s>>>(g, bd, body, c->d_pan_group, c->d_group_start, U, dens, c->d_corr_off,
                                            c->d_corr_j, c->d_corr_val32, c->d_xcorr_off, c->d_xcorr_j,
                                            c->d_xcorr_val32, y);
    PGB_CUDA(cudaGetLastError());
    PGB_LAUNCHED(c, launches);
}

}  // namespace

// The imposed-boundary rows of surface `body` (its current imposed value) into
// y, which the caller has zeroed.
void imposed_rows_f32(pgb_ctx* c, int body, double* y) {
    switch (c->p.P) {
        case 0: run<0>(c, body, y); break;
        case 1: run<1>(c, body, y); break;
        case 2: run<2>(c, body, y); break;
        case 3: run<3>(c, body, y); break;
        case 4: run<4>(c, body, y); break;
        case 5: run<5>(c, body, y); break;
        case 6: run<6>(c, body, y); break;
        case 7: run<7>(c, body, y); break;
        case 8: run<8>(c, body, y); break;
        default: fail(PGB_EINVAL, "the transposed treecode takes P in 0..8");
    }
}

}  // namespace pgb
