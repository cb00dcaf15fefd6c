"""GPU: products and solves of a context that may not keep anything only to be
faster (pgb_keep_limit 0) against those of one that may.  Columns found in the
near lists are the table's to the last bit, so direct sums are too; moments and
near-field sums formed anew are added up in another order."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from problems import gpu_context, spheres  # noqa: E402

import paper_1506_03745_gb300 as pgb  # noqa: E402


def _product(ctx, x, precision):
    xt = torch.tensor(x, device="cuda", dtype=torch.float32 if precision == pgb.PGB_FP32 else torch.float64)
    y = torch.empty_like(xt)
    pgb.pgb_matvec(ctx, xt, y, precision)
    return y.cpu().numpy()


@pytest.mark.parametrize("K,leaf", [(1, 1), (3, 300), (4, 5), (7, 32)])
def test_direct_sums_without_the_column_table_are_the_same_bits(K, leaf):
    bodies = spheres(mol_nu=5, level_srf=2, kind="phi")
    ctx = gpu_context(bodies, theta=0.0, K=K, leaf_size=leaf)
    try:
        x = np.random.default_rng(1).normal(size=pgb.pgb_num_unknowns(ctx))
        want = [_product(ctx, x, p) for p in (pgb.PGB_FP32, pgb.PGB_FP64, pgb.PGB_FP64_DS)]
        assert pgb.pgb_keep_limit(ctx)["columns"] > 0
        assert pgb.pgb_keep_limit(ctx, 0)["columns"] == 0
        with pytest.raises(pgb.PgbError):
            _product(ctx, x, pgb.PGB_FP32)  # the new bound wants a new tree
        pgb.pgb_tree_build(ctx)
        for move in (False, True):
            if move:  # the lists kept, other offsets: there and back
                t = np.array([0.25, 0.0, -0.125])
                for at in (t, np.zeros(3)):
                    pgb.pgb_set_pose(ctx, 0, np.eye(3), at)
                    pgb.pgb_tree_refresh(ctx)
            got = [_product(ctx, x, p) for p in (pgb.PGB_FP32, pgb.PGB_FP64, pgb.PGB_FP64_DS)]
            assert pgb.pgb_keep_limit(ctx, 0) == dict(columns=0, moments=0, near=0)
            for a, b in zip(want, got):
                assert np.array_equal(a, b)
    finally:
        pgb.pgb_destroy(ctx)


@pytest.mark.parametrize("P,K", [(0, 7), (3, 1), (6, 7), (8, 4), (15, 3)])
def test_products_with_nothing_kept(P, K):
    """Sums of some thousand terms in another order: a few hundred roundings."""
    bodies = spheres(level_mol=3, level_srf=3)
    ctx = gpu_context(bodies, P=P, K=K, leaf_size=16)
    try:
        x = np.random.default_rng(2).normal(size=pgb.pgb_num_unknowns(ctx))
        for precision, tol in ((pgb.PGB_FP32, 200 * 2.0 ** -24), (pgb.PGB_FP64, 200 * 2.0 ** -53), (pgb.PGB_FP64_DS, 200 * 2.0 ** -47)):
            a = _product(ctx, x, precision)
            pgb.pgb_keep_limit(ctx, 0)
            pgb.pgb_tree_build(ctx)
            b = _product(ctx, x, precision)
            pgb.pgb_keep_limit(ctx, -1)
            pgb.pgb_tree_build(ctx)
            assert np.linalg.norm(a - b) <= tol * np.linalg.norm(a), precision
    finally:
        pgb.pgb_destroy(ctx)


@pytest.mark.parametrize("mode", [1, 2])
def test_solves_and_batches_with_nothing_kept(mode):
    bodies = spheres(level_mol=2, level_srf=2)
    ctx = gpu_context(bodies, batch=2)
    try:
        x = torch.empty(pgb.pgb_num_unknowns(ctx), dtype=torch.float64, device="cuda")
        R = np.tile(np.eye(3).reshape(9), (2, 1))
        t = np.array([[0.0, 0.0, 0.0], [-0.5, 0.2, 0.0]])
        got = []
        for limit in (-1, 0):
            pgb.pgb_keep_limit(ctx, limit)
            pgb.pgb_set_pose(ctx, 0, np.eye(3), np.zeros(3))
            pgb.pgb_tree_build(ctx)
            code, _ = pgb.pgb_solve(ctx, mode, 1e-9, 500, 100, x)
            assert code == 0
            e = pgb.pgb_energy(ctx, x)["total"]
            code, F, _ = pgb.pgb_solve_batch(ctx, 0, R, t, mode, 1e-9, 500, 100)
            assert code == 0
            got.append([e, *np.asarray(F)[:, 3]])
            if limit == 0:
                assert pgb.pgb_keep_limit(ctx, 0) == dict(columns=0, moments=0, near=0)
            else:
                assert pgb.pgb_keep_limit(ctx)["near"] > 0
        # twice the residual tolerance, amplified by the energy's cancellation of Coulomb terms
        np.testing.assert_allclose(got[0], got[1], rtol=1e-7)
    finally:
        pgb.pgb_destroy(ctx)
