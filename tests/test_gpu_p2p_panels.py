"""GPU: the P2P sums panel by panel (the far rule's points as c and
c - 3 alpha (v_k - c), squared distances from the panel's products) against
the oracle's dense rows by direct summation (theta = 0): every far rule, both
surface kinds, ragged groups and stages, and the smallest work items."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from problems import gpu_context, oracle_system, spheres  # noqa: E402

import paper_1506_03745_gb300 as pgb  # noqa: E402

# |y - A x| <= tol (|A| |x|) row by row.  FP64: its reciprocal square root is
# good to 1e-13, the rest rounds at 1e-16; double-single: near 1e-13 a value.
# FP32: coordinates relative to the group's centre (at most 40 point distances
# away) round at 2^-24, and the distance takes that error |d| / r <= 3 times
# twice over: 240 * 2^-24 = 1.4e-5 an entry.
TOL = {"fp64": 1e-12, "ds": 2e-12, "fp32": 2e-5}
PREC = {"fp64": 1, "ds": 3, "fp32": 0}


@pytest.mark.parametrize("precision", sorted(TOL))
@pytest.mark.parametrize("K", [1, 3, 4, 7])
@pytest.mark.parametrize("kind,nu,level,leaf,item", [("sigma", 3, 1, 32, 64), ("phi", 2, 1, 5, 1), ("sigma", 1, 0, 1, 3)])
def test_direct_sum_matches_dense_rows(precision, K, kind, nu, level, leaf, item):
    bodies = spheres(level_srf=level, kind=kind, mol_nu=nu)
    system = oracle_system(bodies, theta=0.0, K=K)
    A, _ = system.assemble()
    x = np.random.default_rng(7).normal(size=system.n)
    if precision == "fp32":
        x = x.astype(np.float32).astype(np.float64)
    ctx = gpu_context(bodies, theta=0.0, K=K, leaf_size=leaf, p2p_item=item)
    try:
        dt = torch.float32 if precision == "fp32" else torch.float64
        xd = torch.tensor(x, device="cuda", dtype=dt)
        y = torch.empty_like(xd)
        pgb.pgb_matvec(ctx, xd, y, PREC[precision])
        err = np.abs(y.double().cpu().numpy() - A @ x)
        assert (err <= TOL[precision] * (np.abs(A) @ np.abs(x))).all(), (err / (np.abs(A) @ np.abs(x))).max()
    finally:
        pgb.pgb_destroy(ctx)


@pytest.mark.parametrize("mode", ["fp64", "refine"])
@pytest.mark.parametrize("K", [1, 3, 4, 7])
@pytest.mark.parametrize("kind,nu,level,leaf,item", [("sigma", 3, 1, 32, 64), ("phi", 2, 1, 5, 1), ("sigma", 1, 0, 1, 3)])
def test_solve_with_the_kept_near_field_meets_the_dense_rows(mode, K, kind, nu, level, leaf, item):
    """The products of a solve read the near field that its first product
    stored: the solution's residual against the oracle's dense rows is within
    the solver's tolerance plus the operator's own error (TOL above)."""
    bodies = spheres(level_srf=level, kind=kind, mol_nu=nu)
    system = oracle_system(bodies, theta=0.0, K=K)
    A, b = system.assemble()
    ctx = gpu_context(bodies, theta=0.0, K=K, leaf_size=leaf, p2p_item=item)
    try:
        x = torch.empty(system.n, dtype=torch.float64, device="cuda")
        for _ in range(2):  # forming the near field, and with it already there
            code, st = pgb.pgb_solve(ctx, pgb.PGB_FP64 if mode == "fp64" else pgb.PGB_FP32_REFINE, 1e-10, 500, 100, x)
            assert code == 0, st
            xs = x.cpu().numpy()
            off = 4e-12 * np.linalg.norm(np.abs(A) @ np.abs(xs))
            assert np.linalg.norm(A @ xs - b) <= 1e-10 * np.linalg.norm(b) + off
        pgb.pgb_set_pose(ctx, 0, np.eye(3), np.array([-0.5, 0.2, 0.0]))  # other lists: another near field
        pgb.pgb_tree_build(ctx)
        bodies[0].update(R=np.eye(3), t=np.array([-0.5, 0.2, 0.0]))
        A, b = oracle_system(bodies, theta=0.0, K=K).assemble()
        code, st = pgb.pgb_solve(ctx, pgb.PGB_FP64 if mode == "fp64" else pgb.PGB_FP32_REFINE, 1e-10, 500, 100, x)
        xs = x.cpu().numpy()
        assert code == 0, st
        assert np.linalg.norm(A @ xs - b) <= 1e-10 * np.linalg.norm(b) + 4e-12 * np.linalg.norm(np.abs(A) @ np.abs(xs))
    finally:
        pgb.pgb_destroy(ctx)
