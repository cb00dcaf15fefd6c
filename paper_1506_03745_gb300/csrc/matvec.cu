// Treecode matvec driver: source densities, upward pass + evaluation,
// near-field corrections and the block rows of Eq. 6 / Eq. 7.
#include <algorithm>

#include "treecode.cuh"

namespace pgb {

void treecode_launch_f32(int stage, int P, const UpArgs& up, const EvalArgs& ev, const void* xrel, void* mom,
                         const void* far, cudaStream_t s);
void treecode_launch_f64(int stage, int P, const UpArgs& up, const EvalArgs& ev, const void* xrel, void* mom,
                         const void* far, cudaStream_t s);
void treecode_launch_ds(int stage, int P, const UpArgs& up, const EvalArgs& ev, const void* xrel, void* mom,
                        const void* far, cudaStream_t s);
void near_build_f32(const EvalArgs& ev, int K, const void* ng, const void* xrel, void* mat, cudaStream_t s);
void near_build_f64(const EvalArgs& ev, int K, const void* ng, const void* xrel, void* mat, cudaStream_t s);
int64_t near_groups(pgb_ctx* c, void* out);
void convert_pd_ds(const void* pd64, void* pd_ds, int64_t n, cudaStream_t s);

static inline int nblk(int64_t n, int t) { return (int)std::max<int64_t>(1, (n + t - 1) / t); }

// A product's input and output vector: FP64, or the FP32 arrays of an FP32
// product (read and written in place: two launches less than by way of FP64
// copies).
struct VecIn {
    const double* d;
    const float* f;
    __device__ __forceinline__ double operator[](int64_t i) const { return f ? (double)f[i] : d[i]; }
};
struct VecOut {
    double* d;
    float* f;
    __device__ __forceinline__ void put(int64_t i, double v) const {
        if (f) f[i] = (float)v;
        else d[i] = v;
    }
};

// Panel densities (psi_L, psi_Y, phi) of the combined potential U = S_V - S_K
// for every sorted panel (dens), and the same times the panel's area (pd).
//   dielectric: psi_L = dphi, psi_Y = (eps_in/eps_out) dphi, phi = phi
//   imposed potential: psi_Y = u; imposed charge: phi = u
// pd: the panel densities times the area (and wcorr, far_rule_f32_scale, in FP32).
// known == true builds the imposed-boundary densities instead: phi0 as the
// double-layer density of an imposed-potential surface, dphi = -sigma0/eps_out
// as the single layer of an imposed-charge surface, zero on molecules.
// mode 0: densities of the unknowns x; 1: imposed parts only; 2: both (the
// unknowns plus the imposed sigma0 / phi0 of every surface).
template <typename real>
__global__ void k_src_prep(Geo g, BodyDev bd, VecIn x, int mode, typename V4<real>::t* __restrict__ pd, real* __restrict__ dens, double eps_out,
                           double wcorr) {
    const bool known = mode == 1;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= g.n_pan) return;
    const int b = g.pbody[i];
    const int64_t loc = g.perm[i] - bd.pan_off[b];
    const int64_t N = bd.pan_off[b + 1] - bd.pan_off[b];
    const int64_t o = bd.unk_off[b];
    double psiL = 0, psiY = 0, phi = 0;
    const int kind = bd.kind[b];
    if (!known) {
        if (kind == PGB_DIELECTRIC) {
            phi = x[o + loc];
            psiL = x[o + N + loc];
            psiY = bd.eps_ratio[b] * psiL;
        } else if (kind == PGB_SET_POTENTIAL) {
            psiY = x[o + loc];
        } else {
            phi = x[o + loc];
        }
    } else {
        if (kind == PGB_SET_POTENTIAL) phi = bd.bc[b];
        else if (kind == PGB_SET_CHARGE) psiY = -bd.bc[b] / eps_out;
    }
    if (mode == 2) {
        if (kind == PGB_SET_POTENTIAL) phi = bd.bc[b];
        else if (kind == PGB_SET_CHARGE) psiY = -bd.bc[b] / eps_out;
    }
    // the FP32 product keeps its densities in FP32, the FP64 product in FP64
    const real rL = (real)psiL, rY = (real)psiY, rp = (real)phi;
    dens[3 * i] = rL;
    dens[3 * i + 1] = rY;
    dens[3 * i + 2] = rp;
    const real area = (real)(g.A[i] * wcorr);
    typename V4<real>::t pv;
    pv.x = area * rL;
    pv.y = area * rY;
    pv.z = area * rp;
    pv.w = 0;
    pd[i] = pv;
}

// U += near-field corrections (FP64), then the rows of Eq. 6 / Eq. 7 in the
// caller's layout.  mode 0: y = A x.  mode 1: right-hand side of the imposed
// boundary terms, -(U + jump) on exterior and surface rows.  mode 2: the rows
// with the imposed densities included, so that b - A x = b_Coulomb - y.
// Treecode sums of panel i: the partial sums of its group's P2P items, then
// of its M2P items, in item order (a fixed order: the result does not depend
// on the schedule).
struct Parts {
    const int32_t *pan_group, *gstart;
    const int64_t *pitem_off, *fitem_off;
    const double *Up, *Uf;
    int64_t g_lo, g_hi;  // rows of the groups g_lo <= g < g_hi only (a rank's rows of a sharded product)
};

// real: the arithmetic of the near-field corrections (FP32 product: FP32
// copies of the FP64-computed corrections with compensated sums; FP64 product:
// FP64).  ASM_LANES lanes share a panel: they take its correction entries in
// turn (coalesced, seven steps for the usual 25 instead of 25 dependent ones;
// a thread per panel left the GPU at 12 % of its warps, waiting), lane 0 sums
// the group's Laplace partials and writes the interior row, lane 1 the Yukawa
// partials and the exterior or surface row.  2 x 20480 panels: 21 -> 10 us.
#define ASM_LANES 4
template <typename real>
__global__ void __launch_bounds__(128) k_assemble(Geo g, BodyDev bd, Parts u, const real* __restrict__ dens,
                           const int64_t* __restrict__ coff, const int32_t* __restrict__ cj,
                           const typename V4<real>::t* __restrict__ cval, const int64_t* __restrict__ xoff,
                           const int32_t* __restrict__ xj, const typename V4<real>::t* __restrict__ xval, int mode,
                           VecIn x, VecOut y) {
    using v4 = typename V4<real>::t;
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t i = t / ASM_LANES;
    const int sub = (int)(t % ASM_LANES);
    int gi = -1;
    if (i < g.n_pan) gi = u.pan_group[i];
    if (gi < u.g_lo || gi >= u.g_hi) gi = -1;  // (all lanes stay for the exchanges below)
    double s = 0;  // lane 0: Laplace, lane 1: Yukawa
    real c[2] = {0, 0}, e[2] = {0, 0};
    if (gi >= 0) {
        if (sub < 2) {
            const int lane = (int)(i - u.gstart[gi]) + 32 * sub;
            for (int64_t it = u.pitem_off[gi]; it < u.pitem_off[gi + 1]; ++it) s += u.Up[64 * it + lane];
            for (int64_t it = u.fitem_off[gi]; it < u.fitem_off[gi + 1]; ++it) s += u.Uf[64 * it + lane];
        }
        for (int64_t k = coff[i] + sub; k < coff[i + 1]; k += ASM_LANES) {
            const int64_t j = cj[k];
            const v4 d = cval[k];
            const real psiL = dens[3 * j], psiY = dens[3 * j + 1], phi = dens[3 * j + 2];
            if (sizeof(real) == 4) {
                kadd(c[0], e[0], d.x * psiL - d.y * phi);
                kadd(c[1], e[1], d.z * psiY - d.w * phi);
            } else {
                c[0] += d.x * psiL - d.y * phi;
                c[1] += d.z * psiY - d.w * phi;
            }
        }
        for (int64_t k = xoff[i] + sub; k < xoff[i + 1]; k += ASM_LANES) {  // cross-body entries (Yukawa only)
            const int64_t j = xj[k];
            const v4 d = xval[k];
            if (sizeof(real) == 4) kadd(c[1], e[1], d.z * dens[3 * j + 1] - d.w * dens[3 * j + 2]);
            else c[1] += d.z * dens[3 * j + 1] - d.w * dens[3 * j + 2];
        }
    }
#pragma unroll
    for (int o = ASM_LANES / 2; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const real oc = __shfl_xor_sync(0xffffffffu, c[q], o);
            if (sizeof(real) == 4) {
                e[q] += __shfl_xor_sync(0xffffffffu, e[q], o);
                kadd(c[q], e[q], oc);
            } else {
                c[q] += oc;
            }
        }
    if (gi < 0 || sub > 1) return;
    const double U = s * (1.0 / PGB_FOUR_PI) + ((double)c[sub] + (double)e[sub]);
    const int b = g.pbody[i];
    const int64_t loc = g.perm[i] - bd.pan_off[b];
    const int64_t N = bd.pan_off[b + 1] - bd.pan_off[b];
    const int64_t o = bd.unk_off[b];
    const int kind = bd.kind[b];
    if (sub == 0) {  // interior row (no imposed terms: Laplace couples a body only to itself)
        if (kind == PGB_DIELECTRIC && mode != 1) y.put(o + loc, 0.5 * x[o + loc] - U);
    } else if (mode == 1) {
        if (kind == PGB_DIELECTRIC) y.put(o + N + loc, -U);
        else y.put(o + loc, kind == PGB_SET_CHARGE ? -U : -(U + 0.5 * bd.bc[b]));
    } else {
        // the jump terms from the unknowns themselves, in FP64
        if (kind == PGB_DIELECTRIC) y.put(o + N + loc, 0.5 * x[o + loc] + U);
        else if (kind == PGB_SET_CHARGE) y.put(o + loc, U + 0.5 * x[o + loc]);
        else y.put(o + loc, U + (mode == 2 ? 0.5 * bd.bc[b] : 0.0));  // jump of the imposed phi0
    }
}

// ---------------------------------------------------------------- nested interfaces
// With nested interfaces every row is its body's jump term minus the
// representation sum of the region the row belongs to (the interior row of a
// dielectric body: its interior; the exterior row, or a surface's row: the
// region around it), and each region's sum runs as its own treecode pass.
// Rows start from the jump terms (modes 0 and 2; mode 1: minus the imposed
// jump).
__global__ void k_rows_init(Geo g, BodyDev bd, const double* x, int mode, double* y) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= g.n_pan) return;
    const int b = g.pbody[i];
    const int64_t loc = g.perm[i] - bd.pan_off[b];
    const int64_t N = bd.pan_off[b + 1] - bd.pan_off[b];
    const int64_t o = bd.unk_off[b];
    const int kind = bd.kind[b];
    if (kind == PGB_DIELECTRIC) {
        const double v = mode == 1 ? 0.0 : 0.5 * x[o + loc];
        y[o + loc] = v;
        y[o + N + loc] = v;
    } else if (kind == PGB_SET_CHARGE) {
        y[o + loc] = mode == 1 ? 0.0 : 0.5 * x[o + loc];
    } else {
        y[o + loc] = mode == 0 ? 0.0 : (mode == 2 ? 0.5 * bd.bc[b] : -0.5 * bd.bc[b]);
    }
}

// Panel densities of one region's pass: every body on the region's boundary
// with the densities of its side of the interface and the side's sign folded
// in, so that the pass sums s [V psi - K phi] (the Yukawa slots, at the
// region's screening; kappa = 0 is Laplace); all other bodies are zero.
//   dielectric: phi, psi = fac dphi (fac = 1 inside, eps_in / eps_R outside)
//   imposed potential: psi = u, phi = phi0 (known); imposed charge: phi = u,
//   psi = -sigma0 / eps_R (known).   mode as k_src_prep (x unused for 1).
template <typename real>
__global__ void k_src_region(Geo g, BodyDev bd, RegionDev rd, const double* __restrict__ x, int mode,
                             typename V4<real>::t* __restrict__ pd, real* __restrict__ dens, double wcorr) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= g.n_pan) return;
    const int b = g.pbody[i];
    const int sg = rd.sign[b];
    double psi = 0, phi = 0;
    if (sg != 0) {
        const int64_t loc = g.perm[i] - bd.pan_off[b];
        const int64_t N = bd.pan_off[b + 1] - bd.pan_off[b];
        const int64_t o = bd.unk_off[b];
        const int kind = bd.kind[b];
        if (kind == PGB_DIELECTRIC) {
            if (mode != 1) {
                phi = x[o + loc];
                psi = rd.fac[b] * x[o + N + loc];
            }
        } else if (kind == PGB_SET_POTENTIAL) {
            if (mode != 1) psi = x[o + loc];
            if (mode != 0) phi = bd.bc[b];
        } else {
            if (mode != 1) phi = x[o + loc];
            if (mode != 0) psi = rd.psi_known[b];
        }
        psi *= sg;
        phi *= sg;
    }
    const real rY = (real)psi, rp = (real)phi;
    dens[3 * i] = 0;
    dens[3 * i + 1] = rY;
    dens[3 * i + 2] = rp;
    const real area = (real)(g.A[i] * wcorr);
    typename V4<real>::t pv;
    pv.x = 0;
    pv.y = area * rY;
    pv.z = area * rp;
    pv.w = 0;
    pd[i] = pv;
}

// One region's sums into its rows: the pass's item partials (Yukawa slots)
// plus the region's near-field corrections, subtracted from the row of the
// target's side (added for mode 1, the right-hand side of imposed terms).
template <typename real>
__global__ void k_assemble_region(Geo g, BodyDev bd, RegionDev rd, Parts u, const real* __restrict__ dens,
                                  const int64_t* __restrict__ coff, const int32_t* __restrict__ cj,
                                  const typename V4<real>::t* __restrict__ cval, const int64_t* __restrict__ xoff,
                                  const int32_t* __restrict__ xj, const typename V4<real>::t* __restrict__ xval,
                                  int mode, double* __restrict__ y) {
    using v4 = typename V4<real>::t;
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= g.n_pan) return;
    const int b = g.pbody[i];
    const int sg = rd.sign[b];
    if (sg == 0) return;
    const int gi = u.pan_group[i];
    if (gi < u.g_lo || gi >= u.g_hi) return;
    const int lane = (int)(i - u.gstart[gi]);
    double sY = 0;
    for (int64_t it = u.pitem_off[gi]; it < u.pitem_off[gi + 1]; ++it) sY += u.Up[64 * it + 32 + lane];
    for (int64_t it = u.fitem_off[gi]; it < u.fitem_off[gi + 1]; ++it) sY += u.Uf[64 * it + 32 + lane];
    double U = sY * (1.0 / PGB_FOUR_PI);
    real cY = 0, eY = 0;
    for (int64_t e = coff[i]; e < coff[i + 1]; ++e) {
        const int64_t j = cj[e];
        const v4 d = cval[e];
        if (sizeof(real) == 4) kadd(cY, eY, d.z * dens[3 * j + 1] - d.w * dens[3 * j + 2]);
        else cY += d.z * dens[3 * j + 1] - d.w * dens[3 * j + 2];
    }
    for (int64_t e = xoff[i]; e < xoff[i + 1]; ++e) {
        const int64_t j = xj[e];
        const v4 d = xval[e];
        if (sizeof(real) == 4) kadd(cY, eY, d.z * dens[3 * j + 1] - d.w * dens[3 * j + 2]);
        else cY += d.z * dens[3 * j + 1] - d.w * dens[3 * j + 2];
    }
    U += (double)cY + (double)eY;
    const int64_t loc = g.perm[i] - bd.pan_off[b];
    const int64_t N = bd.pan_off[b + 1] - bd.pan_off[b];
    const int64_t o = bd.unk_off[b];
    const int64_t r = (bd.kind[b] == PGB_DIELECTRIC && sg < 0) ? o + N + loc : o + loc;
    y[r] += mode == 1 ? U : -U;
}

__global__ void k_f32_to_f64(const float* a, double* b, int64_t n) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) b[i] = a[i];
}
__global__ void k_f64_to_f32(const double* a, float* b, int64_t n) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) b[i] = (float)a[i];
}
void convert_f32_f64(const float* a, double* b, int64_t n, cudaStream_t s) {
    k_f32_to_f64<<<nblk(n, 256), 256, 0, s>>>(a, b, n);
}
void convert_f64_f32(const double* a, float* b, int64_t n, cudaStream_t s) {
    k_f64_to_f32<<<nblk(n, 256), 256, 0, s>>>(a, b, n);
}

static void apply_vec(pgb_ctx* c, VecIn xv, VecOut yv, int precision, int mode, const int* known_mask);

void apply_operator(pgb_ctx* c, const double* x, double* y, int precision, bool known_only, const int* known_mask) {
    apply_mode(c, x, y, precision, known_only ? 1 : 0, known_mask);
}

void apply_full(pgb_ctx* c, const double* x, double* y, int precision) { apply_mode(c, x, y, precision, 2, nullptr); }

// One stage of the treecode in the arithmetic `kind` (0 FP32, 1 FP64, 2
// double-single).
static void launch_stage(pgb_ctx* c, int stage, int kind, const UpArgs& up, const EvalArgs& ev, void* mom,
                         cudaStream_t s) {
    if (kind == 0) treecode_launch_f32(stage, c->p.P, up, ev, c->d_x32, mom, up.far, s);
    else if (kind == 1) treecode_launch_f64(stage, c->p.P, up, ev, c->d_x64, mom, up.far, s);
    else treecode_launch_ds(stage, c->p.P, up, ev, c->d_x64, mom, up.far, s);
}

int sm_count(pgb_ctx* c) {
    if (!c->sms) {
        int dev = 0;
        PGB_CUDA(cudaGetDevice(&dev));
        PGB_CUDA(cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev));
    }
    return c->sms;
}

size_t keep_bound(pgb_ctx* c, int share) {
    if (c->keep_limit >= 0) return (size_t)c->keep_limit;
    if (!c->dev_bytes) {
        size_t free_b = 0;
        PGB_CUDA(cudaMemGetInfo(&free_b, &c->dev_bytes));
    }
    return c->dev_bytes / share;
}

// The panel moments of the current geometry in the arithmetic `kind`: formed on
// the context's stream the first time a product of that kind meets the
// geometry, kept until the geometry or the order changes.  nullptr where they
// would take more than a sixteenth of the device's memory (336 bytes a panel in
// FP32 at order 6, 3.3 KB at order 15) or cannot be allocated: the P2M then
// forms them on the spot.
const void* panel_moments(pgb_ctx* c, int kind) {
    auto& pm = c->pan_mom[kind];
    if (pm.geom_gen == c->geom_gen && pm.P == c->p.P) return pm.have ? (const void*)pm.buf.p : nullptr;
    if (c->capturing) return nullptr;  // (every product is prepared outside the capture)
    // the caller captures: what is launched now runs when its graph does, and
    // products before that need moments too
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    PGB_CUDA(cudaStreamIsCapturing(c->stream, &cs));
    if (cs != cudaStreamCaptureStatusNone) return nullptr;
    pm.have = false;
    pm.geom_gen = c->geom_gen;
    pm.P = c->p.P;
    const size_t esz = kind == 0 ? 4 : 8;
    const size_t bytes = (size_t)c->n_pan * n_terms(c->p.P) * esz;
    if (bytes > keep_bound(c, 16)) {
        pm.buf.release();
        return nullptr;
    }
    try {
        pm.buf.resize(bytes);
    } catch (const Error& e) {
        if (e.code != PGB_ENOMEM) throw;
        return nullptr;
    }
    UpArgs up = {};
    up.sms = sm_count(c);
    up.K = c->p.K;
    up.rule = far_rule(c->p.K);
    up.pg = kind == 0 ? (const void*)c->d_pg32.p : kind == 1 ? (const void*)c->d_pg64.p : (const void*)c->d_pg_ds.p;
    EvalArgs ev = {};
    ev.n_pan = c->n_pan;
    StageTimer tm(c, PGB_STAGE_UPWARD + (kind == 0 ? 0 : PGB_STAGE_FP64));
    launch_stage(c, STAGE_PANEL_MOMENTS, kind, up, ev, pm.buf.p, c->stream);
    PGB_CUDA(cudaGetLastError());
    PGB_LAUNCHED(c, 1);
    pm.have = true;
    return pm.buf.p;
}

// Memory a stream-ordered allocation can have: what the device has free and what
// the device's pool holds unused.
static size_t free_bytes() {
    size_t free_b = 0, total_b = 0;
    PGB_CUDA(cudaMemGetInfo(&free_b, &total_b));
    int dev = 0;
    cudaMemPool_t pool;
    uint64_t held = 0, used = 0;
    PGB_CUDA(cudaGetDevice(&dev));
    PGB_CUDA(cudaDeviceGetDefaultMemPool(&pool, dev));
    PGB_CUDA(cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &held));
    PGB_CUDA(cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used));
    return free_b + (held > used ? held - used : 0);
}

// Gives the stored near fields back to the pool: all of them (the lists change),
// or those that take more than a 32nd of their bound (a solve has ended; 1.1 GB
// here, what 150000 panels hold in FP32 -- forming one anew is a few hundredths of
// the next solve).
void near_release(pgb_ctx* c, bool large_only) {
    for (auto& nm : c->near_mat) {
        const size_t bound = c->keep_limit >= 0 ? (size_t)c->keep_limit : c->dev_bytes / 8;
        if (!nm.buf.p || (large_only && nm.buf.n <= bound / 32)) continue;
        if (nm.buf.st != c->stream) cudaStreamSynchronize(c->stream);  // (freed in the order of its own stream)
        nm.buf.release();
        nm.list_gen = ~0ull;
    }
}

// The stored near field of the current lists for a product of a running solve
// (NearScope): formed by the solve's first product on the context's stream, at
// about the cost of one P2P, and kept until the lists, the geometry
// or the screening change.  Not kept (the P2P then forms the sums, as products
// outside solves do) where it would take more than an eighth of the device's
// memory or a quarter of what is free, or cannot be allocated.
bool near_ready(pgb_ctx* c, int kind) {
    auto& nm = c->near_mat[kind];
    if (nm.list_gen == c->list_gen && nm.kappa == c->kappa) return nm.have;
    if (c->capturing) return false;  // (every product is prepared outside the capture)
    nm.have = false;
    nm.list_gen = c->list_gen;
    nm.kappa = c->kappa;
    if (c->n_groups == 0 || c->n_pitems == 0 || !c->d_col.p) return false;
    try {
        nm.group.resize(16 * c->n_groups);
        const int64_t units = near_groups(c, nm.group.p);
        const size_t bytes = (size_t)units * 64 * (kind == 0 ? 4 : 8);
        if (bytes > nm.buf.n) {
            nm.buf.release();
            if (bytes > keep_bound(c, 8) || bytes > free_bytes() / 4) return false;
            nm.buf.resize(bytes);
        }
    } catch (const Error& e) {
        if (e.code != PGB_ENOMEM) throw;
        return false;
    }
    EvalArgs ev = {};
    ev.gstart = c->d_group_start;
    ev.gend = c->d_group_end;
    ev.gcenter = c->d_group_center;
    ev.ncenter = c->d_node_center;
    ev.kappa = c->kappa;
    ev.col_off = c->d_col_off;
    ev.col = c->d_col;
    ev.pnode = c->d_pnode;
    ev.rule = far_rule(c->p.K);
    ev.n_pitems = c->n_pitems;
    ev.pitem_off = c->d_pitem_off;
    ev.pitem_group = c->d_pitem_group;
    ev.pg = kind == 0 ? (const void*)c->d_pg32.p : (const void*)c->d_pg64.p;
    StageTimer tm(c, PGB_STAGE_P2P + (kind == 0 ? 0 : PGB_STAGE_FP64));
    if (kind == 0) near_build_f32(ev, c->p.K, nm.group.p, c->d_x32, nm.buf.p, c->stream);
    else near_build_f64(ev, c->p.K, nm.group.p, c->d_x64, nm.buf.p, c->stream);
    PGB_CUDA(cudaGetLastError());
    PGB_LAUNCHED(c, 1);
    nm.have = true;
    return true;
}

// Upward pass as a CUDA graph: captured (on a private stream; nothing runs
// there) the first time a tree / buffer / source-activity combination is
// used, then one cudaGraphLaunch on the context stream per product.
static void upward_graph(pgb_ctx* c, int kind, const UpArgs& up, const EvalArgs& ev, void* mom, cudaStream_t on) {
    auto& gr = c->up_graph[kind];
    bool ok = gr.exec && gr.tree_gen == c->tree_gen && gr.pd == up.pd && gr.pg == up.pg && gr.pmom == up.pmom &&
              gr.mom == mom && gr.ncenter == up.ncenter &&
              gr.p2m_grid == up.p2m_grid && gr.far == up.far && gr.far_tab == up.far_tab;
    for (int b = 0; ok && b < PGB_MAX_BODIES; ++b) ok = gr.src_active[b] == up.src_active[b];
    if (!ok) {
        if (gr.exec) {
            PGB_CUDA(cudaGraphExecDestroy(gr.exec));
            gr.exec = nullptr;
        }
        if (!c->cap_stream) PGB_CUDA(cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking));
        PGB_CUDA(cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeThreadLocal));
        std::string why;
        try {
            launch_stage(c, PGB_STAGE_UPWARD, kind, up, ev, mom, c->cap_stream);
        } catch (const Error& e) {
            why = e.msg;
        }
        const cudaError_t le = cudaGetLastError();
        cudaGraph_t graph = nullptr;
        const cudaError_t ce = cudaStreamEndCapture(c->cap_stream, &graph);
        if (!why.empty() || le != cudaSuccess || ce != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            (void)cudaGetLastError();
            fail(PGB_ECUDA, "upward-pass graph capture: " + (why.empty() ? std::string(cudaGetErrorString(
                                                                               le != cudaSuccess ? le : ce))
                                                                          : why));
        }
        const cudaError_t ie = cudaGraphInstantiate(&gr.exec, graph, 0);
        cudaGraphDestroy(graph);
        if (ie != cudaSuccess) gr.exec = nullptr;
        PGB_CUDA(ie);
        gr.tree_gen = c->tree_gen;
        gr.pd = up.pd;
        gr.pg = up.pg;
        gr.pmom = up.pmom;
        gr.mom = mom;
        gr.far = up.far;
        gr.far_tab = up.far_tab;
        gr.ncenter = up.ncenter;
        gr.p2m_grid = up.p2m_grid;
        for (int b = 0; b < PGB_MAX_BODIES; ++b) gr.src_active[b] = up.src_active[b];
    }
    PGB_CUDA(cudaGraphLaunch(gr.exec, on));
}

// The upward-pass stream of a precision (created on first use).
static cudaStream_t upward_stream(pgb_ctx* c, int pi) {
    if (!c->up_stream[pi]) {
        int least = 0, greatest = 0;
        PGB_CUDA(cudaDeviceGetStreamPriorityRange(&least, &greatest));
        PGB_CUDA(cudaStreamCreateWithPriority(&c->up_stream[pi], cudaStreamNonBlocking, greatest));
        PGB_CUDA(cudaEventCreateWithFlags(&c->up_fork[pi], cudaEventDisableTiming));
        PGB_CUDA(cudaEventCreateWithFlags(&c->up_join[pi], cudaEventDisableTiming));
    }
    return c->up_stream[pi];
}

// Sizes every buffer a product of this precision writes (so that a product
// on another stream allocates nothing).
void reserve_product(pgb_ctx* c, int precision) {
    const int pi = precision == PGB_FP32 ? 0 : 1;
    const int T = n_terms(c->p.P);
    c->d_dens[pi].resize(3 * c->n_pan);
    c->d_Up[pi].resize(64 * std::max<int64_t>(c->n_pitems, 1));
    c->d_Uf[pi].resize(64 * std::max<int64_t>(c->n_fitems, 1));
    c->d_work.resize(2);
    const int TP = n_far_pad(c->p.P);
    if (pi == 0) {
        c->d_pd32.resize(c->n_pan);
        c->d_mom32.resize((size_t)c->n_nodes * 2 * T);
        c->d_far32.resize((size_t)c->n_nodes * 2 * TP);
    } else {
        c->d_pd64.resize(c->n_pan);
        c->d_pd_ds.resize(c->n_pan);
        c->d_mom64.resize((size_t)c->n_nodes * 2 * T);
        c->d_far64.resize((size_t)c->n_nodes * 2 * TP);
        c->d_mom_ds.resize((size_t)c->n_nodes * 2 * T);
        c->d_far_ds.resize((size_t)c->n_nodes * 2 * TP);
    }
    (void)panel_moments(c, precision == PGB_FP32 ? 0 : precision == PGB_FP64_DS ? 2 : 1);
    (void)far_table(c, c->kappa);
    for (const auto& reg : c->regions) (void)far_table(c, reg->dev.kappa);
    if (c->arrive_gen[pi] != c->tree_gen || c->d_arrive[pi].n < (size_t)c->n_nodes) {
        c->d_arrive[pi].resize(std::max<int64_t>(c->n_nodes, 1));
        PGB_CUDA(cudaMemsetAsync(c->d_arrive[pi].p, 0, sizeof(int) * c->d_arrive[pi].n, c->stream));
        c->arrive_gen[pi] = c->tree_gen;
    }
}

void apply_mode(pgb_ctx* c, const double* x, double* y, int precision, int mode, const int* known_mask) {
    apply_vec(c, VecIn{x, nullptr}, VecOut{y, nullptr}, precision, mode, known_mask);
}

void apply_f32(pgb_ctx* c, const float* x, float* y) {
    if (!nested(c)) {
        apply_vec(c, VecIn{nullptr, x}, VecOut{nullptr, y}, PGB_FP32, 0, nullptr);
        return;
    }
    c->d_xtmp.resize(c->n_unk);
    c->d_ytmp.resize(c->n_unk);
    convert_f32_f64(x, c->d_xtmp, c->n_unk, c->stream);
    apply_mode(c, c->d_xtmp, c->d_ytmp, PGB_FP32, 0, nullptr);
    convert_f64_f32(c->d_ytmp, y, c->n_unk, c->stream);
}

static void apply_vec(pgb_ctx* c, VecIn xv, VecOut yv, int precision, int mode, const int* known_mask) {
    const double* x = xv.d;
    double* y = yv.d;
    const bool known_only = mode == 1;
    if (!c->tree_valid) fail(PGB_ESTATE, "pgb_tree_build has not run for the current bodies and poses");
    cudaStream_t s = c->stream;
    Geo g = geo(c);
    BodyDev bd = body_dev(c);
    if (known_only && known_mask)  // imposed terms of the selected surfaces only
        for (int b = 0; b < bd.n_bodies; ++b)
            if (!known_mask[b]) bd.bc[b] = 0.0;
    const int P = c->p.P;
    const int T = n_terms(P);
    // per-precision work buffers: an FP64 product may run on a side stream
    // while FP32 products go on
    const int pi = precision == PGB_FP32 ? 0 : 1;
    auto& dens = c->d_dens[pi];
    auto& Up = c->d_Up[pi];
    auto& Uf = c->d_Uf[pi];
    dens.resize(3 * c->n_pan);
    Up.resize(64 * std::max<int64_t>(c->n_pitems, 1));
    Uf.resize(64 * std::max<int64_t>(c->n_fitems, 1));
    UpArgs up;
    up.n_leaves = c->n_leaves;
    up.leaf_node = c->d_leaf_node; up.nstart = c->d_node_start; up.nend = c->d_node_end;
    up.child = c->d_node_child; up.nchild = c->d_node_nchild;
    up.ncenter = c->d_node_center; up.K = c->p.K; up.nbody = c->d_node_body;
    up.sms = sm_count(c);
    up.p2m_grid = 0;
    up.n_nodes = c->n_nodes;
    up.parent = c->d_node_parent;
    up.n_internal = c->n_nodes - c->n_leaves;
    up.internal_node = c->d_internal_node;
    up.n_ichild = c->d_node_nichild;
    {
        const int pi_up = precision == PGB_FP32 ? 0 : 1;
        auto& cnt = c->d_arrive[pi_up];
        if (c->arrive_gen[pi_up] != c->tree_gen || cnt.n < (size_t)c->n_nodes) {
            cnt.resize(std::max<int64_t>(c->n_nodes, 1));
            PGB_CUDA(cudaMemsetAsync(cnt.p, 0, sizeof(int) * cnt.n, s));
            c->arrive_gen[pi_up] = c->tree_gen;
        }
        up.arrive = cnt.p;
    }
    if (precision != PGB_FP32 && c->persist_blocks > 0)  // side product: P2M on two blocks per SM
        up.p2m_grid = 2 * c->persist_blocks;
    EvalArgs ev;
    ev.n_pan = c->n_pan;
    ev.gstart = c->d_group_start; ev.gend = c->d_group_end; ev.gbody = c->d_group_body;
    ev.gcenter = c->d_group_center; ev.near_off = c->d_near_off; ev.far_off = c->d_far_off;
    ev.near_l = c->d_near; ev.far_l = c->d_far; ev.nstart = c->d_node_start; ev.nend = c->d_node_end;
    ev.nbody = c->d_node_body; ev.ncenter = c->d_node_center; ev.K = c->p.K; ev.kappa = c->kappa;
    for (int b = 0; b < PGB_MAX_BODIES; ++b) ev.lap_body[b] = ev.src_active[b] = up.src_active[b] = 0;
    for (size_t b = 0; b < c->bodies.size(); ++b) {
        ev.lap_body[b] = c->bodies[b].kind == PGB_DIELECTRIC;
        // imposed-boundary terms: molecules carry no known density
        ev.src_active[b] = up.src_active[b] =
            !c->body_off[b] && (known_only ? (known_mask ? known_mask[b] : (c->bodies[b].kind != PGB_DIELECTRIC)) : 1);
    }
    ev.all_active = 1;
    for (size_t b = 0; b < c->bodies.size(); ++b) ev.all_active &= ev.src_active[b];
    // a replayed lockstep iteration: which problems take part is known on the device only
    ev.bmask = up.bmask = c->dev_bmask;
    if (c->dev_bmask) ev.all_active = 0;
    // rows of bodies left out of the product (a lockstep batch's finished
    // problems) are not computed
    ev.tgt_mask = ~0ull;
    for (size_t b = 0; b < c->bodies.size(); ++b)
        if (c->body_off[b]) ev.tgt_mask &= ~(1ull << b);
    ev.g_lo = c->shard_g[0] >= 0 ? c->shard_g[0] : 0;
    ev.g_hi = c->shard_g[0] >= 0 ? c->shard_g[1] : c->n_groups;
    ev.far4 = c->d_far4;
    ev.col_off = c->d_col_off;
    ev.col = c->d_col;
    ev.ent_col = c->d_ent_col;
    ev.cen = c->d_c;
    ev.pnode = c->d_pnode;
    ev.pbody = c->d_pbody;
    ev.pts = c->d_y64;
    ev.rule = far_rule(c->p.K);
    ev.src_mask = 0;
    for (size_t b = 0; b < c->bodies.size(); ++b) ev.src_mask |= (unsigned long long)(ev.src_active[b] != 0) << b;
    ev.n_pitems = c->n_pitems;
    ev.n_fitems = c->n_fitems;
    ev.pitem_off = c->d_pitem_off;
    ev.fitem_off = c->d_fitem_off;
    ev.pitem_group = c->d_pitem_group;
    ev.fitem_group = c->d_fitem_group;
    ev.Up = Up;
    ev.Uf = Uf;
    ev.p2p_work = ev.m2p_work = nullptr;
    ev.persist_blocks = 0;
    if (c->persist_blocks > 0) {  // side-stream product: a few resident blocks per SM take items
        c->d_work.resize(2);
        PGB_CUDA(cudaMemsetAsync(c->d_work.p, 0, 16, s));
        ev.p2p_work = c->d_work.p;
        ev.m2p_work = c->d_work.p + 1;
        ev.persist_blocks = c->persist_blocks;
    }
    const bool f32 = precision == PGB_FP32;
    const double wcorr = f32 ? far_rule_f32_scale(c->p.K) : 1.0;
    const int TP = n_far_pad(P);
    if (f32) {
        c->d_pd32.resize(c->n_pan);
        c->d_mom32.resize((size_t)c->n_nodes * 2 * T);
        c->d_far32.resize((size_t)c->n_nodes * 2 * TP);
        up.far = c->d_far32.p;
        ev.pg = c->d_pg32.p;
        ev.pd = c->d_pd32.p;
    } else {
        c->d_pd64.resize(c->n_pan);
        c->d_mom64.resize((size_t)c->n_nodes * 2 * T);
        c->d_far64.resize((size_t)c->n_nodes * 2 * TP);
        up.far = c->d_far64.p;
        ev.pg = c->d_pg64.p;
        ev.pd = c->d_pd64.p;
        if (precision == PGB_FP64_DS) {
            c->d_pd_ds.resize(c->n_pan);
            c->d_mom_ds.resize((size_t)c->n_nodes * 2 * T);
            c->d_far_ds.resize((size_t)c->n_nodes * 2 * TP);
            up.far = c->d_far_ds.p;
        }
    }
    const bool dsp = precision == PGB_FP64_DS;
    const int kind = f32 ? 0 : dsp ? 2 : 1;
    void* mom = f32 ? (void*)c->d_mom32.p : dsp ? (void*)c->d_mom_ds.p : (void*)c->d_mom64.p;
    up.rule = ev.rule;
    up.pg = dsp ? (const void*)c->d_pg_ds.p : ev.pg;
    up.pd = dsp ? (const void*)c->d_pd_ds.p : ev.pd;
    up.pmom = panel_moments(c, kind);
    if (kind < 2 && ((c->near_on >> kind) & 1) && !ev.p2p_work && c->shard_g[0] < 0 && !nested(c) && near_ready(c, kind)) {
        ev.near_mat = c->near_mat[kind].buf.p;
        ev.near_group = c->near_mat[kind].group.p;
    }
    auto tab_for = [&](double kappa) -> const void* {
        const FarTab& t = far_table(c, kappa);
        if (f32) return t.t32.p;
        return dsp ? (const void*)t.tds.p : (const void*)t.t64.p;
    };
    up.far_tab = tab_for(c->kappa);
    if (nested(c)) {
        // one treecode pass per region: rows from the jump terms, then each
        // region's sum subtracted from the rows on its boundary
        if (known_mask) fail(PGB_EINVAL, "imposed-term selection is not available with nested interfaces");
        k_rows_init<<<nblk(c->n_pan, 128), 128, 0, s>>>(g, bd, x, mode, y);
        PGB_LAUNCHED(c, 1);
        for (int b = 0; b < PGB_MAX_BODIES; ++b) ev.lap_body[b] = 0;
        for (const auto& reg : c->regions) {
            const RegionDev& rd = reg->dev;
            ev.kappa = rd.kappa;
            up.far_tab = tab_for(rd.kappa);
            if (ev.p2p_work)  // persistent launches take items from counters: fresh ones per pass
                PGB_CUDA(cudaMemsetAsync(c->d_work.p, 0, 16, s));
            ev.all_active = 1;
            ev.tgt_mask = 0;
            ev.src_mask = 0;
            for (size_t b = 0; b < c->bodies.size(); ++b) {
                ev.src_active[b] = up.src_active[b] = rd.sign[b] != 0 && !c->body_off[b];
                ev.all_active &= ev.src_active[b];
                if (ev.src_active[b]) {  // only the region's own rows
                    ev.tgt_mask |= 1ull << b;
                    ev.src_mask |= 1ull << b;
                }
            }
            {
                StageTimer tm(c, PGB_STAGE_SOURCES + (f32 ? 0 : PGB_STAGE_FP64));
                if (f32)
                    k_src_region<float><<<nblk(c->n_pan, 128), 128, 0, s>>>(g, bd, rd, x, mode, c->d_pd32,
                                                                             (float*)dens.p, wcorr);
                else
                    k_src_region<double><<<nblk(c->n_pan, 128), 128, 0, s>>>(g, bd, rd, x, mode, c->d_pd64,
                                                                              dens.p, wcorr);
                if (precision == PGB_FP64_DS) convert_pd_ds(c->d_pd64, c->d_pd_ds, c->n_pan, s);
                PGB_CUDA(cudaGetLastError());
                PGB_LAUNCHED(c, precision == PGB_FP64_DS ? 2 : 1);
            }
            for (int stage : {PGB_STAGE_UPWARD, PGB_STAGE_P2P, PGB_STAGE_M2P}) {
                StageTimer tm(c, stage + (f32 ? 0 : PGB_STAGE_FP64));
                launch_stage(c, stage, kind, up, ev, mom, s);
                PGB_CUDA(cudaGetLastError());
                PGB_LAUNCHED(c, stage == PGB_STAGE_UPWARD ? 3 : 1);
            }
            {
                StageTimer tm(c, PGB_STAGE_ASSEMBLE + (f32 ? 0 : PGB_STAGE_FP64));
                Parts u{c->d_pan_group, c->d_group_start, c->d_pitem_off, c->d_fitem_off, Up, Uf, ev.g_lo, ev.g_hi};
                if (f32)
                    k_assemble_region<float><<<nblk(c->n_pan, 128), 128, 0, s>>>(
                        g, bd, rd, u, (const float*)dens.p, reg->corr_off, reg->corr_j, reg->corr_val32,
                        reg->xcorr_off, reg->xcorr_j, reg->xcorr_val32, mode, y);
                else
                    k_assemble_region<double><<<nblk(c->n_pan, 128), 128, 0, s>>>(
                        g, bd, rd, u, dens.p, reg->corr_off, reg->corr_j, reg->corr_val, reg->xcorr_off, reg->xcorr_j,
                        reg->xcorr_val, mode, y);
                PGB_CUDA(cudaGetLastError());
                PGB_LAUNCHED(c, 1);
            }
        }
        return;
    }
    {
        StageTimer tm(c, PGB_STAGE_SOURCES + (f32 ? 0 : PGB_STAGE_FP64));
        if (f32)
            k_src_prep<float><<<nblk(c->n_pan, 128), 128, 0, s>>>(g, bd, xv, mode, c->d_pd32,
                                                                  (float*)dens.p, c->eps_out, wcorr);
        else
            k_src_prep<double><<<nblk(c->n_pan, 128), 128, 0, s>>>(g, bd, xv, mode, c->d_pd64,
                                                                   dens.p, c->eps_out, wcorr);
        if (precision == PGB_FP64_DS) convert_pd_ds(c->d_pd64, c->d_pd_ds, c->n_pan, s);
        PGB_CUDA(cudaGetLastError());
        PGB_LAUNCHED(c, precision == PGB_FP64_DS ? 2 : 1);
    }
    // the upward pass on its own stream, beside P2P (which does not read the
    // moments)
    cudaStream_t us = upward_stream(c, pi);
    PGB_CUDA(cudaEventRecord(c->up_fork[pi], s));
    PGB_CUDA(cudaStreamWaitEvent(us, c->up_fork[pi], 0));
    {
        StageTimer tm(c, PGB_STAGE_UPWARD + (f32 ? 0 : PGB_STAGE_FP64), us);
        if (c->p.graphs && !c->capturing) {
            upward_graph(c, kind, up, ev, mom, us);
            c->graph_kernels += 3;
            ++c->graph_launches;
        } else {
            launch_stage(c, PGB_STAGE_UPWARD, kind, up, ev, mom, us);
        }
        PGB_CUDA(cudaGetLastError());
        PGB_LAUNCHED(c, 3);
    }
    // M2P follows the upward pass on its stream: the two evaluations write
    // different sums, and what one leaves idle at its end the other uses
    // (2 x 20480 panels: 18 us less for the product)
    for (int stage : {PGB_STAGE_M2P, PGB_STAGE_P2P}) {
        cudaStream_t on = stage == PGB_STAGE_M2P ? us : s;
        StageTimer tm(c, stage + (f32 ? 0 : PGB_STAGE_FP64), on);
        launch_stage(c, stage, kind, up, ev, mom, on);
        PGB_CUDA(cudaGetLastError());
        PGB_LAUNCHED(c, 1);
    }
    PGB_CUDA(cudaEventRecord(c->up_join[pi], us));
    PGB_CUDA(cudaStreamWaitEvent(s, c->up_join[pi], 0));
    {
        StageTimer tm(c, PGB_STAGE_ASSEMBLE + (f32 ? 0 : PGB_STAGE_FP64));
        Parts u{c->d_pan_group, c->d_group_start, c->d_pitem_off, c->d_fitem_off, Up, Uf, ev.g_lo, ev.g_hi};
        if (f32)
            k_assemble<float><<<nblk(ASM_LANES * c->n_pan, 128), 128, 0, s>>>(
                g, bd, u, (const float*)dens.p, c->d_corr_off, c->d_corr_j, c->d_corr_val32, c->d_xcorr_off,
                c->d_xcorr_j, c->d_xcorr_val32, mode, xv, yv);
        else
            k_assemble<double><<<nblk(ASM_LANES * c->n_pan, 128), 128, 0, s>>>(g, bd, u, dens.p, c->d_corr_off, c->d_corr_j,
                                                                   c->d_corr_val, c->d_xcorr_off, c->d_xcorr_j,
                                                                   c->d_xcorr_val, mode, xv, yv);
        PGB_CUDA(cudaGetLastError());
        PGB_LAUNCHED(c, 1);
    }
}

}  // namespace pgb
