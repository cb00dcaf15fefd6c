"""GPU: how far double-single products round from FP64 ones, as direct sums, so
that nothing but P2P differs.

The bounds are what sums point by point with Newton's and Taylor's forms of
1/sqrt and 2^x showed on the same inputs (relative, 2-norm).  Points of a panel
that share the rounding of its distance and normal product lie 2.6e-15 to
4.9e-15 off and miss all of them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from problems import gpu_context, spheres, star_molecule  # noqa: E402

import paper_1506_03745_gb300 as pgb  # noqa: E402


@pytest.mark.parametrize("kappa", [0.125, 0.0])
@pytest.mark.parametrize("which,K,bound", [("spheres", 1, 1.47e-15), ("spheres", 7, 1.20e-15), ("star", 1, 3.68e-15),
                                           ("star", 7, 2.90e-15)])
def test_direct_sum_rounds_no_further_than_point_by_point(which, K, bound, kappa):
    bodies = spheres(mol_nu=8, level_srf=3) if which == "spheres" else star_molecule(nu=10)
    ctx = gpu_context(bodies, kappa=kappa, theta=0.0, K=K)
    try:
        x = torch.tensor(np.random.default_rng(1).normal(size=pgb.pgb_num_unknowns(ctx)), device="cuda")
        y64, yds = torch.empty_like(x), torch.empty_like(x)
        pgb.pgb_matvec(ctx, x, y64, pgb.PGB_FP64)
        pgb.pgb_matvec(ctx, x, yds, pgb.PGB_FP64_DS)
        off = float(torch.linalg.norm(yds - y64) / torch.linalg.norm(y64))
        assert off <= bound, off
    finally:
        pgb.pgb_destroy(ctx)
