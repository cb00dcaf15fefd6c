"""GPU: the FP64 transposed product in the harmonic basis and the stored near
field read the other way (gradients), over far rules, orders and ragged
leaves, against the forward product and the dense oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.gradient import gradients  # noqa: E402
from problems import gpu_context, oracle_system, spheres  # noqa: E402

import paper_1506_03745_gb300 as pgb  # noqa: E402


@pytest.mark.parametrize("P", [0, 1, 2, 5, 8])
@pytest.mark.parametrize("K,leaf,item", [(1, 3, 64), (3, 8, 1), (4, 32, 5), (7, 13, 64)])
def test_transposed_product_is_the_transpose(P, K, leaf, item):
    """<A x, lam> = <x, A^T lam>: both sides sum the same terms, each good to
    1e-13 (the reciprocal square root), a row's near and far terms cancelling
    by at most 100."""
    bodies = spheres(level_srf=3, kind="sigma", mol_nu=5)
    ctx = gpu_context(bodies, theta=0.6, P=P, K=K, leaf_size=leaf, m2p_item=item)
    try:
        assert pgb.pgb_tree_stats(ctx)["n_far"] > 0
        n = pgb.pgb_num_unknowns(ctx)
        rng = np.random.default_rng(3)
        x, lam = (torch.tensor(v, device="cuda") for v in rng.normal(size=(2, n)))
        y, yt = torch.empty_like(x), torch.empty_like(x)
        pgb.pgb_matvec(ctx, x, y, pgb.PGB_FP64)
        pgb.pgb_matvec_transpose(ctx, lam, yt, pgb.PGB_FP64)
        scale = max(float(lam.norm() * y.norm()), float(x.norm() * yt.norm()))
        assert abs(float(lam @ y) - float(x @ yt)) <= 1e-11 * scale
    finally:
        pgb.pgb_destroy(ctx)


@pytest.mark.parametrize("kind,K,leaf", [("sigma", 1, 3), ("phi", 3, 32), ("sigma", 4, 7), ("phi", 7, 20)])
def test_gradient_from_the_stored_near_field(kind, K, leaf):
    """Direct sum: the gradient's products all read the stored near field; both
    solves stop at 1e-11 and the systems' condition is below 1e3."""
    bodies = spheres(level_srf=1, kind=kind, mol_nu=3)
    ref = gradients(oracle_system(bodies, theta=0.0, K=K))
    ctx = gpu_context(bodies, theta=0.0, K=K, leaf_size=leaf)
    try:
        x = torch.empty(pgb.pgb_num_unknowns(ctx), dtype=torch.float64, device="cuda")
        code, _ = pgb.pgb_solve(ctx, pgb.PGB_FP64, 1e-11, 3000, 100, x)
        assert code == 0
        code, dq, dbc, dt, _ = pgb.pgb_grad(ctx, x, 1, 2, pgb.PGB_FP64, 1e-11, 3000, 100)
        assert code == 0
        np.testing.assert_allclose(dq, ref["dq"][0], rtol=1e-8, atol=1e-10)
        assert dbc[1] == pytest.approx(ref["dbc"][1], rel=1e-8)
    finally:
        pgb.pgb_destroy(ctx)
