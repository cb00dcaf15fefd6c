"""The work that programs built on this library have it do, as cases to be measured.

Four kinds, each through the package's entry points:

* ``product``  -- one application of the boundary-element operator (``pgb_matvec``), the inner
  step of every Krylov method a program writes around the library, in FP32, FP64 or
  double-single arithmetic;
* ``solve``    -- a new molecule beside a surface: octree, interaction lists and near field from
  the mesh (``pgb_tree_reset`` + ``pgb_tree_build``), the GMRES solve and the energies;
* ``poses``    -- several rigid poses of a molecule beside a surface, solved as one batch
  (``pgb_solve_batch``), the unit of an orientation sweep;
* ``gradient`` -- forward and backward through the autograd wrapper (``FreeEnergy``): tree,
  solve, energy, adjoint solve and the derivatives in charges, imposed values and translations.

A molecule is a closed star-shaped surface r = r0 (1 + smooth random bumps) (``bumps`` 0: a
sphere) meshed as a geodesic sphere of frequency ``nu`` (20 nu^2 panels), with ``nq`` charges
inside; the surface is a geodesic sphere of radius ``rs`` and frequency ``ns`` (0: none) that
holds a charge density ("sigma", C/m^2) or a potential ("phi", V), ``gap`` Angstrom away.
"""
import functools
import math

import numpy as np
import torch

import paper_1506_03745_gb300 as pgb
from paper_1506_03745_gb300.autograd import FreeEnergy

EPS_IN, EPS_OUT = 4.0, 80.0
MAX_ITER, RESTART = 2000, 100
PRECISION = {"fp32": pgb.PGB_FP32, "fp64": pgb.PGB_FP64, "ds": pgb.PGB_FP64_DS}
MODE = {"fp32": pgb.PGB_FP32, "fp64": pgb.PGB_FP64, "refine": pgb.PGB_FP32_REFINE}

# The benchmark's numerical parameters: 7-point far rule, 19-point close-by rule, 9 points per
# edge, Taylor order 6, theta 0.5, 32 panels per leaf.
BASE = dict(nu=32, bumps=0.0, r0=4.0, nq=1, ns=32, rs=4.0, surface="sigma", bc=0.05, gap=4.0, kappa=0.125,
            K=7, K_near=19, P=6, theta=0.5, leaf=32)
# The differentiation and pose workloads: a 15 A molecule with many charges beside a 40 A sphere.
PROTEIN = dict(BASE, nu=17, bumps=0.05, r0=15.0, nq=900, ns=39, rs=40.0, bc=-0.05, gap=10.0)


def case(name, kind, base=BASE, **kw):
    return dict(base, name=name, kind=kind, **kw)


def listed():
    return [
        # the smallest call: coarse meshes, where launches and latency count
        case("product small", "product", nu=4, ns=4, precision="fp32"),
        # the benchmark's operator: the inner product of most solves
        case("product", "product", precision="fp32"),
        # a fine mesh that fills the GPU many times over
        case("product large", "product", nu=101, ns=101, precision="fp32"),
        # the FP64-class product of iterative refinement, on a molecule beside a large sphere (uneven sizes)
        case("product ds", "product", PROTEIN, precision="ds"),
        # the plain FP64 product, a molecule alone
        case("product fp64", "product", PROTEIN, nu=15, ns=0, precision="fp64"),
        # the parameters of the paper's grid-convergence study: order 15, 3-point rule, 300 panels per leaf, held potential
        case("product order 15", "product", r0=5.0, surface="phi", bc=180.95, gap=3.0, K=3, K_near=37, P=15, leaf=300,
             precision="fp32"),
        # the benchmark's step: everything from the mesh to the energies
        case("solve", "solve", mode="refine", tol=1e-11, precond=0),
        # a protein-sized molecule and its charges in salt-free water, held potential, preconditioned
        case("solve protein", "solve", PROTEIN, nu=25, ns=25, kappa=0.0, surface="phi", bc=0.05, mode="refine", tol=1e-11,
             precond=1),
        # a small system in FP64 throughout, as the reference for a study
        case("solve fp64", "solve", PROTEIN, nu=7, ns=9, nq=60, mode="fp64", tol=1e-10, precond=0),
        # a stretch of an orientation sweep near the charged sphere
        case("poses", "poses", PROTEIN, nu=16, ns=21, poses=8, mode="refine", tol=1e-11, precond=1),
        # differentiation of the free energy, forward and backward, with an FP32 adjoint ...
        case("gradient", "gradient", PROTEIN, mode="refine", tol=1e-11, grad="fp32", grad_tol=1e-5),
        # ... and a smaller one in FP64
        case("gradient fp64", "gradient", PROTEIN, nu=10, ns=13, mode="refine", tol=1e-11, grad="fp64", grad_tol=1e-10),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["product"] * 4 + ["solve"] * 3 + ["poses", "gradient"])
    base = PROTEIN if kind in ("poses", "gradient") or rng.random() < 0.5 else BASE
    c = dict(base, kind=kind, kappa=rng.choice([0.125, 0.125, 0.0, round(rng.uniform(0.02, 0.3), 3)]),
             gap=round(rng.uniform(4.0, 14.0), 2))
    if rng.random() < 0.4:
        c.update(surface="phi", bc=0.05)
    order = rng.choice([4, 5, 6, 6, 6, 7, 8])
    c.update(P=order, theta=rng.choice([0.4, 0.5, 0.5, 0.6, 0.7]), leaf=rng.choice([16, 24, 32, 32, 48, 64]),
             K=rng.choice([3, 4, 7, 7, 7]))
    if base is PROTEIN:
        c["nq"] = log(20, 900)
    if kind == "product":
        c["precision"] = rng.choice(["fp32", "fp32", "fp32", "ds", "fp64"])
        top = {"fp32": 90, "ds": 40, "fp64": 16}[c["precision"]]
        c.update(nu=log(4, top), ns=log(4, top) if rng.random() < 0.75 else 0)
        if c["precision"] == "fp32" and rng.random() < 0.25:
            c.update(P=rng.choice([10, 12, 15]), K=3, K_near=37, leaf=rng.choice([100, 200, 300]))
    elif kind == "solve":
        c["mode"] = rng.choice(["refine", "refine", "refine", "fp64"])
        top = 32 if c["mode"] == "refine" else 9
        c.update(nu=log(5, top), ns=log(5, top) if rng.random() < 0.75 else 0, tol=1e-11, precond=rng.choice([0, 1]))
    elif kind == "poses":
        c.update(nu=log(6, 16), ns=log(6, 21), poses=rng.randint(2, 8), mode="refine", tol=1e-11, precond=rng.choice([0, 1]))
    else:
        # the adjoint wants the bodies farther apart than twice a panel's size
        c.update(nu=log(6, 10), ns=rng.randint(11, 13), gap=round(rng.uniform(9.0, 14.0), 2), mode="refine", tol=1e-11,
                 grad=rng.choice(["fp32", "fp64"]))
        c["grad_tol"] = 1e-5 if c["grad"] == "fp32" else 1e-10
    return c


# ---------------------------------------------------------------- inputs

@functools.lru_cache(maxsize=8)
def _geodesic(nu):
    """Unit geodesic sphere: every icosahedron face cut into nu^2 triangles."""
    g = (1.0 + math.sqrt(5.0)) / 2.0
    v = np.array([[-1, g, 0], [1, g, 0], [-1, -g, 0], [1, -g, 0], [0, -1, g], [0, 1, g], [0, -1, -g], [0, 1, -g],
                  [g, 0, -1], [g, 0, 1], [-g, 0, -1], [-g, 0, 1]])
    v /= np.linalg.norm(v[0])
    f = np.array([[0, 11, 5], [0, 5, 1], [0, 1, 7], [0, 7, 10], [0, 10, 11], [1, 5, 9], [5, 11, 4], [11, 10, 2],
                  [10, 7, 6], [7, 1, 8], [3, 9, 4], [3, 4, 2], [3, 2, 6], [3, 6, 8], [3, 8, 9], [4, 9, 5], [2, 4, 11],
                  [6, 2, 10], [8, 6, 7], [9, 8, 1]])
    i, j = np.meshgrid(np.arange(nu + 1), np.arange(nu + 1), indexing="ij")
    keep = i + j <= nu
    i, j = i[keep], j[keep]
    at = -np.ones((nu + 2, nu + 2), dtype=np.int64)
    at[i, j] = np.arange(len(i))
    bary = np.stack([i, j, nu - i - j], 1) / nu
    up = (i + j < nu)
    down = (i + j < nu - 1)
    tri = np.concatenate([
        np.stack([at[i[up], j[up]], at[i[up] + 1, j[up]], at[i[up], j[up] + 1]], 1),
        np.stack([at[i[down] + 1, j[down]], at[i[down] + 1, j[down] + 1], at[i[down], j[down] + 1]], 1)])
    pts = np.einsum("kb,fbx->fkx", bary, v[f]).reshape(-1, 3)
    pts /= np.linalg.norm(pts, axis=1, keepdims=True)
    tris = (tri[None] + len(i) * np.arange(20)[:, None, None]).reshape(-1, 3)
    _, first, same = np.unique(np.round(pts * 1e8).astype(np.int64), axis=0, return_index=True, return_inverse=True)
    pts, tris = pts[first], same.reshape(-1)[tris]
    a, b, c = (pts[tris[:, k]] for k in range(3))
    turned = np.einsum("ij,ij->i", np.cross(b - a, c - a), a + b + c) < 0
    tris[turned] = tris[turned][:, [0, 2, 1]]
    return pts, tris.astype(np.int32)


def _rotations(rng, n):
    q = rng.normal(size=(n, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                     2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                     2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).reshape(n, 3, 3)


def _bodies(c, rng):
    """The molecule (posed so that its closest vertex is `gap` from the surface) and the surface."""
    u, f = _geodesic(c["nu"])
    shape = np.ones(len(u))
    if c["bumps"]:
        for _ in range(12):
            shape += c["bumps"] * rng.normal() * np.cos(u @ (2.0 * rng.normal(size=3)) + rng.uniform(0, 2 * math.pi)) / 2
        shape = np.maximum(shape, 0.6)
    v = c["r0"] * u * shape[:, None]
    if c["nq"] == 1:
        xyz, q = np.zeros((1, 3)), np.array([rng.uniform(0.5, 1.5)])
    else:
        d = rng.normal(size=(c["nq"], 3))
        d *= ((0.9 * c["r0"] * shape.min() * rng.random(c["nq"]) ** (1 / 3)) / np.linalg.norm(d, axis=1))[:, None]
        xyz, q = d, rng.uniform(-0.8, 0.8, c["nq"])
    R = _rotations(rng, 1)[0]
    mol = dict(kind=pgb.PGB_DIELECTRIC, verts=v, tris=f, xyz=xyz, q=q, bc=0.0, R=R, t=np.zeros(3))
    if not c["ns"]:
        return [mol]
    us, fs = _geodesic(c["ns"])
    mol["t"] = _placed(v, R, c["rs"], c["gap"])
    kind = pgb.PGB_SET_CHARGE if c["surface"] == "sigma" else pgb.PGB_SET_POTENTIAL
    return [mol, dict(kind=kind, verts=us * c["rs"], tris=fs, xyz=np.zeros((0, 3)), q=np.zeros(0),
                      bc=c["bc"] * rng.uniform(0.8, 1.2), R=_rotations(rng, 1)[0], t=np.zeros(3))]


def _placed(v, R, rs, gap):
    """Translation along x that leaves `gap` between the rotated vertices v and the sphere rs at the origin."""
    w = v @ R.T
    d2 = np.maximum((rs + gap) ** 2 - w[:, 1] ** 2 - w[:, 2] ** 2, 0.0)
    return np.array([np.max(np.where(d2 > 0, np.sqrt(d2) - w[:, 0], -np.inf)), 0.0, 0.0])


class _Context:
    """Owns a pgb context, as a program's handle class does."""

    def __init__(self, c, bodies, **params):
        self.handle = pgb.pgb_create(pgb.default_params(K=c["K"], K_near=c["K_near"], P=c["P"], theta=c["theta"],
                                                        leaf_size=c["leaf"], **params), torch.cuda.current_stream())
        for i, b in enumerate(bodies):
            has = len(b["q"]) > 0
            pgb.pgb_mesh_load(self.handle, b["kind"], b["verts"], b["tris"], EPS_IN, b["xyz"] if has else None,
                              b["q"] if has else None, b["bc"])
            pgb.pgb_set_pose(self.handle, i, b["R"], b["t"])
        pgb.pgb_set_solvent(self.handle, EPS_OUT, c["kappa"])

    def __del__(self):
        if getattr(self, "handle", None) is not None:
            torch.cuda.current_stream().synchronize()
            pgb.pgb_destroy(self.handle)


def _pose_set(c, bodies, rng):
    R = _rotations(rng, c["poses"])
    gaps = c["gap"] + np.resize([-4.0, -2.0, 0.0, 4.0], c["poses"])
    return R, np.stack([_placed(bodies[0]["verts"], R[k], c["rs"], max(3.0, gaps[k])) for k in range(len(R))])


def prepare(c, seed):
    rng = np.random.default_rng([seed, 1506])
    bodies = _bodies(c, rng)
    s = dict(case=c, bodies=bodies)
    if c["kind"] == "product":
        s["ctx"] = _Context(c, bodies)
        pgb.pgb_tree_build(s["ctx"].handle)
        n = pgb.pgb_num_unknowns(s["ctx"].handle)
        dtype = torch.float32 if c["precision"] == "fp32" else torch.float64
        g = torch.Generator(device="cuda").manual_seed(seed)
        s["x"] = torch.randn(n, generator=g, device="cuda", dtype=torch.float64).to(dtype)
        s["y"] = torch.empty(n, device="cuda", dtype=dtype)
    elif c["kind"] == "solve":
        s["ctx"] = _Context(c, bodies, precond=c["precond"])
        n = pgb.pgb_num_unknowns(s["ctx"].handle)
        s["x"] = torch.zeros(n, device="cuda", dtype=torch.float64)
    elif c["kind"] == "poses":
        s["ctx"] = _Context(c, bodies, precond=c["precond"], batch=c["poses"])
        s["R"], s["t"] = _pose_set(c, bodies, rng)
    else:
        s["ctx"] = _Context(c, bodies)
        s["fe"] = FreeEnergy(s["ctx"].handle, [b["kind"] for b in bodies], [len(b["q"]) for b in bodies],
                             R=[b["R"] for b in bodies], mode=MODE[c["mode"]], tol=c["tol"],
                             grad_precision=PRECISION[c["grad"]], grad_tol=c["grad_tol"])
        s["q"] = torch.tensor(bodies[0]["q"], requires_grad=True)
        s["bc"] = torch.tensor([b["bc"] for b in bodies], dtype=torch.float64, requires_grad=True)
        s["at"] = torch.tensor(np.array([b["t"] for b in bodies]), requires_grad=True)
    return s


def run(s):
    c = s["case"]
    h = s["ctx"].handle
    if c["kind"] == "product":
        pgb.pgb_matvec(h, s["x"], s["y"], PRECISION[c["precision"]])
        return s["y"]
    if c["kind"] == "solve":
        pgb.pgb_tree_reset(h)
        pgb.pgb_tree_build(h)
        pgb.pgb_solve(h, MODE[c["mode"]], c["tol"], MAX_ITER, RESTART, s["x"])
        return {"x": s["x"], "energies": pgb.pgb_energy(h, s["x"])}
    if c["kind"] == "poses":
        _, F, _ = pgb.pgb_solve_batch(h, 0, s["R"], s["t"], MODE[c["mode"]], c["tol"], MAX_ITER, RESTART)
        return F
    for p in (s["q"], s["bc"], s["at"]):
        p.grad = None
    F = s["fe"](s["q"], s["bc"], s["at"])
    F.backward()
    return {"F": F, "q": s["q"].grad, "bc": s["bc"].grad, "t": s["at"].grad}


# ---------------------------------------------------------------- work

def work(c):
    """Counted from the sizes: a target of the treecode meets about 4.5 leaf / theta^2 panels point by
    point (at most every panel) and 35 / theta^2 nodes through expansions, which is what the benchmark's
    lists hold; 29 operations a (target, point), 4 a coefficient and target.  A solve counts 40 products."""
    N, S = 20 * c["nu"] ** 2, 20 * c["ns"] ** 2
    n = N + S
    near = min(n, 4.5 * c["leaf"] / c["theta"] ** 2) * c["K"]
    far = 35 / c["theta"] ** 2 if n > near / c["K"] else 0
    terms = (c["P"] + 1) * (c["P"] + 2) * (c["P"] + 3) / 6
    product = n * (29 * near + far * 4 * terms)
    mesh = 36.0 * n + 32.0 * c["nq"]
    unknowns = 2 * N + S
    if c["kind"] == "product":
        return {"bytes": mesh + 2 * unknowns * (4 if c["precision"] == "fp32" else 8), "flops": product}
    if c["kind"] == "solve":
        return {"bytes": mesh + 8 * unknowns, "flops": 40 * product}
    if c["kind"] == "poses":
        return {"bytes": mesh + 128.0 * c["poses"], "flops": 40 * c["poses"] * product}
    return {"bytes": mesh + 8.0 * (c["nq"] + 8), "flops": 80 * product}


# ---------------------------------------------------------------- 64-bit values

E_CHARGE, EPS0 = 1.602176634e-19, 8.8541878128e-12
KCAL = E_CHARGE ** 2 / (EPS0 * 1e-10) * 6.02214076e23 / 4184.0
PER_C_M2, PER_VOLT = 1e-20 / E_CHARGE, EPS0 * 1e-10 / E_CHARGE
FOUR_PI = 4.0 * math.pi
DENSE_UNKNOWNS, DIRECT_PANELS = 13000, 50000


def _orbits(centre, three, six):
    """Barycentric points and weights of a symmetric rule: the centroid's weight, (a, w) for the points
    (a, a, 1 - 2a) and (a, b, w) for the six permutations of (a, b, 1 - a - b)."""
    pts, w = ([[1 / 3] * 3], [centre]) if centre else ([], [])
    for a, wt in three:
        pts += [[a, a, 1 - 2 * a], [a, 1 - 2 * a, a], [1 - 2 * a, a, a]]
        w += [wt] * 3
    for a, b, wt in six:
        d = 1 - a - b
        pts += [[a, b, d], [b, a, d], [a, d, b], [d, a, b], [b, d, a], [d, b, a]]
        w += [wt] * 6
    return np.array(pts), np.array(w)


ROOT15 = math.sqrt(15.0)
TRI = {
    1: _orbits(1.0, [], []),
    3: _orbits(0, [(1 / 6, 1 / 3)], []),
    4: _orbits(-0.5625, [(0.2, 25 / 48)], []),
    7: _orbits(0.225, [((6 + ROOT15) / 21, (155 + ROOT15) / 1200), ((6 - ROOT15) / 21, (155 - ROOT15) / 1200)], []),
    # degree 9 (19 points) and degree 13 (37 points), fully symmetric
    19: _orbits(0.097135796282798836, [(0.48968251919999046, 0.031334700227139071), (0.43708959149478511, 0.077827541004774279),
                                       (0.18820353561957844, 0.079647738927210249), (0.044729513394400086, 0.025577675658698031)],
                [(0.036838412054976998, 0.22196298916048389, 0.043283539377289376)]),
    37: _orbits(0.067960036586246178, [(0.22137228629077266, 0.058278485119104967),
                                     (0.48907694645276972, 0.023994401928280732),
                                     (0.021509681108241863, 0.0060523371032162624),
                                     (0.42694141425852916, 0.055601967530146151)],
                [(0.024370186900963597, 0.86470777029809476, 0.014965401104833563),
                 (0.27251581777159456, 0.72235779312635251, 0.0095906810035390009),
                 (0.068012243553901175, 0.62354599554840595, 0.034641276140611924),
                 (0.16359740107118323, 0.74850711589943242, 0.024179039812933768)]),
}


class _Panels:
    def __init__(self, b, c, dev):
        put = functools.partial(torch.as_tensor, dtype=torch.float64, device=dev)
        world = b["verts"] @ b["R"].T + b["t"]
        self.v = put(world[b["tris"]])
        self.c = self.v.mean(1)
        cr = torch.linalg.cross(self.v[:, 1] - self.v[:, 0], self.v[:, 2] - self.v[:, 0])
        nr = cr.norm(dim=1)
        self.n, self.A, self.N = cr / nr[:, None], 0.5 * nr, len(nr)
        self.rules = []
        for k in (c["K"], c["K_near"]):
            pts, w = TRI[k]
            self.rules.append((torch.einsum("kb,nbx->knx", put(pts), self.v), put(w)[:, None] * self.A))
        self.q, self.xyz = put(b["q"]), put(b["xyz"] @ b["R"].T + b["t"]) if len(b["q"]) else put(b["xyz"])
        self.kind = b["kind"]
        self.bc = b["bc"] * {pgb.PGB_DIELECTRIC: 0.0, pgb.PGB_SET_CHARGE: PER_C_M2, pgb.PGB_SET_POTENTIAL: PER_VOLT}[b["kind"]]


def _point(d, n, w, kappa):
    r2 = (d * d).sum(-1)
    r = torch.where(r2 > 0, r2, torch.ones_like(r2)).sqrt()
    on = (r2 > 0).to(r.dtype) * w / FOUR_PI
    nd = (n * d).sum(-1)
    vl = on / r
    kl = vl * nd / (r * r)
    e = torch.exp(-kappa * r)
    return vl, kl, vl * e, kl * e * (1 + kappa * r)


def _entries(x, own, p, kappa):
    """V_L, K_L, V_Y, K_Y (targets x panels): the point rule of each distance, the panel's own integral in closed
    form along its edges.  own: index of the target's own panel, or None."""
    out = [0.0] * 4
    for y, w in zip(*p.rules[0]):
        out = [o + g for o, g in zip(out, _point(x[:, None] - y[None], p.n[None], w[None], kappa))]
    near = ((x[:, None] - p.c[None]) ** 2).sum(-1) < 8 * p.A[None]
    rows = torch.arange(len(x), device=x.device)
    if own is not None:
        near[rows, own] = False
    i, j = near.nonzero(as_tuple=True)
    fine = [0.0] * 4
    for y, w in zip(*p.rules[1]):
        fine = [o + g for o, g in zip(fine, _point(x[i] - y[j], p.n[j], w[j], kappa))]
    for o, g in zip(out, fine):
        o[i, j] = g
    if own is not None:
        s, w = np.polynomial.legendre.leggauss(9)
        vl = vy = 0.0
        for a in range(3):
            pa, pb, c = p.v[own, a], p.v[own, (a + 1) % 3], x
            e = pb - pa
            ell = e.norm(dim=1)
            h = torch.linalg.cross(c - pa, e).norm(dim=1) / ell
            for sk, wk in zip((s + 1) / 2, w / 2):
                rho = (pa + sk * e - c).norm(dim=1)
                jac = h / rho ** 2 * ell * wk / FOUR_PI
                vl = vl + rho * jac
                vy = vy + ((1 - torch.exp(-kappa * rho)) / kappa if kappa > 0 else rho) * jac
        for o, g in zip(out, (vl, 0.0, vy, 0.0)):
            o[rows, own] = g
    return out


def _offsets(ps):
    o = [0]
    for p in ps:
        o.append(o[-1] + (2 if p.kind == pgb.PGB_DIELECTRIC else 1) * p.N)
    return o


def _rows(ps, kappa, a, lo, hi, use):
    """Calls use(row index, column offset, block) for the operator's rows of panels lo:hi of body a."""
    off, p = _offsets(ps), ps[a]
    ext = off[a] + (p.N if p.kind == pgb.PGB_DIELECTRIC else 0)
    own = torch.arange(lo, hi, device=p.c.device)
    for b, q in enumerate(ps):
        vl, kl, vy, ky = _entries(p.c[lo:hi], own if a == b else None, q, kappa)
        half = torch.zeros_like(vl)
        if a == b:
            half[own - lo, own] = 0.5
        if q.kind == pgb.PGB_DIELECTRIC:
            if a == b:
                use(off[a] + lo, off[b], half + kl)
                use(off[a] + lo, off[b] + q.N, -vl)
            use(ext + lo, off[b], half - ky)
            use(ext + lo, off[b] + q.N, EPS_IN / EPS_OUT * vy)
        elif q.kind == pgb.PGB_SET_POTENTIAL:
            use(ext + lo, off[b], vy)
            use(ext + lo, -1, (half - ky).sum(1) * -q.bc)
        else:
            use(ext + lo, off[b], half - ky)
            use(ext + lo, -1, vy.sum(1) * (q.bc / EPS_OUT))


def _each_row(ps, kappa, use):
    step = max(1, (1 << 26) // max(p.N for p in ps))
    for a, p in enumerate(ps):
        for lo in range(0, p.N, step):
            _rows(ps, kappa, a, lo, min(p.N, lo + step), use)


def _system(ps, kappa):
    n = _offsets(ps)[-1]
    A = torch.zeros(n, n, dtype=torch.float64, device=ps[0].c.device)
    b = A.new_zeros(n)

    def use(row, col, block):
        if col < 0:
            b[row:row + len(block)] += block
        else:
            A[row:row + block.shape[0], col:col + block.shape[1]] = block

    _each_row(ps, kappa, use)
    known = b.clone()
    for o, p in zip(_offsets(ps), ps):
        if len(p.q):
            b[o:o + p.N] += (p.q / (FOUR_PI * EPS_IN * torch.cdist(p.c, p.xyz))).sum(1)
    return A, b, known


def _coulomb(p, q):
    if len(p.xyz) < 2:
        return 0.0 * q.sum()
    r = (p.xyz[:, None] - p.xyz[None]).norm(dim=-1) + torch.diag(torch.full((len(q),), math.inf, device=q.device, dtype=q.dtype))
    return 0.5 * (q[:, None] * q[None] / (FOUR_PI * EPS_IN * r)).sum()


def _energies(ps, kappa, x, charge=None, bc=None):
    """Coulomb, solvation and surface energy, in internal units."""
    e = [0.0, 0.0, 0.0]
    for i, (o, p) in enumerate(zip(_offsets(ps), ps)):
        if p.kind == pgb.PGB_DIELECTRIC:
            q = p.q if charge is None else charge
            vl, kl, _, _ = _entries(p.xyz, None, p, kappa)
            e[0] = e[0] + _coulomb(p, q)
            e[1] = e[1] + 0.5 * (q @ (vl @ x[o + p.N:o + 2 * p.N] - kl @ x[o:o + p.N]))
        else:
            beta = (p.bc if bc is None else bc[i]) * (1.0 if p.kind == pgb.PGB_SET_CHARGE else EPS_OUT)
            e[2] = e[2] + 0.5 * beta * (x[o:o + p.N] @ p.A)
    return e


def _gradient(ps, kappa):
    """Free energy and its derivatives in the charges, the imposed values and the translations (adjoint)."""
    A, b, known = _system(ps, kappa)
    x = torch.linalg.solve(A, b)
    xg = x.clone().requires_grad_(True)
    F = sum(_energies(ps, kappa, xg))
    (g,) = torch.autograd.grad(F, xg)
    lam = torch.linalg.solve(A.T, g)
    q = ps[0].q.clone().requires_grad_(True)
    bc = torch.tensor([p.bc for p in ps], dtype=torch.float64, device=x.device, requires_grad=True)
    L = sum(_energies(ps, kappa, x, q, bc)) + lam[:ps[0].N] @ (q / (FOUR_PI * EPS_IN * torch.cdist(ps[0].c, ps[0].xyz))).sum(1)
    dq, dbc = torch.autograd.grad(L, (q, bc))
    dt = torch.zeros(len(ps), 3, dtype=torch.float64, device=x.device)
    if len(ps) == 2:
        dbc[1] += lam @ known / ps[1].bc
        off = _offsets(ps)
        for a, b_ in ((0, 1), (1, 0)):
            p, s = ps[a], ps[b_]
            w = lam[off[a] + p.N:off[a + 1]] if p.kind == pgb.PGB_DIELECTRIC else lam[off[a]:off[a + 1]]
            if s.kind == pgb.PGB_DIELECTRIC:
                phi, psi = x[off[b_]:off[b_] + s.N], EPS_IN / EPS_OUT * x[off[b_] + s.N:off[b_ + 1]]
            elif s.kind == pgb.PGB_SET_CHARGE:
                phi, psi = x[off[b_]:off[b_ + 1]], torch.full((s.N,), -s.bc / EPS_OUT, dtype=torch.float64, device=x.device)
            else:
                phi, psi = torch.full((s.N,), s.bc, dtype=torch.float64, device=x.device), x[off[b_]:off[b_ + 1]]
            shift = torch.zeros(3, dtype=torch.float64, device=x.device, requires_grad=True)
            for lo in range(0, p.N, 256):
                u = 0.0
                for y, wt in zip(*s.rules[0]):
                    _, _, vy, ky = _point(p.c[lo:lo + 256, None] + shift - y[None], s.n[None], wt[None], kappa)
                    u = u + vy @ psi - ky @ phi
                (gr,) = torch.autograd.grad(w[lo:lo + 256] @ u, shift)
                dt[a] -= gr
                dt[b_] += gr
    unit = torch.tensor([0.0] + [PER_C_M2 if p.kind == pgb.PGB_SET_CHARGE else PER_VOLT for p in ps[1:]], dtype=torch.float64,
                        device=x.device)
    return {"F": F.detach() * KCAL, "q": dq * KCAL, "bc": dbc * unit * KCAL, "t": dt * KCAL}


def exact(c, seed):
    rng = np.random.default_rng([seed, 1506])
    bodies = _bodies(c, rng)
    N, S = 20 * c["nu"] ** 2, 20 * c["ns"] ** 2
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if c["kind"] == "product":
        if N + S > DIRECT_PANELS:
            return None
        ps = [_Panels(b, c, dev) for b in bodies]
        g = torch.Generator(device=dev).manual_seed(seed)
        x = torch.randn(_offsets(ps)[-1], generator=g, device=dev, dtype=torch.float64)
        x = x.float().double() if c["precision"] == "fp32" else x
        y = torch.zeros_like(x)

        def use(row, col, block):
            if col >= 0:
                y[row:row + block.shape[0]] += block @ x[col:col + block.shape[1]]

        _each_row(ps, c["kappa"], use)
        return y
    if 2 * N + S > DENSE_UNKNOWNS:
        return None
    if c["kind"] == "poses":
        R, t = _pose_set(c, bodies, rng)
        F = []
        for k in range(c["poses"]):
            bodies[0].update(R=R[k], t=t[k])
            F.append(_solved([_Panels(b, c, dev) for b in bodies], c["kappa"])[1])
        return np.array([[e["coulomb"], e["solvation"], e["surface"], e["total"]] for e in F])
    ps = [_Panels(b, c, dev) for b in bodies]
    if c["kind"] == "solve":
        x, e = _solved(ps, c["kappa"])
        return {"x": x, "energies": e}
    return _gradient(ps, c["kappa"])


def _solved(ps, kappa):
    A, b, _ = _system(ps, kappa)
    x = torch.linalg.solve(A, b)
    e = [float(v) * KCAL for v in _energies(ps, kappa, x)]
    return x, dict(coulomb=e[0], solvation=e[1], surface=e[2], total=sum(e))
