"""GPU: which near fields a context holds (pgb_keep_limit reports the bytes)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from problems import gpu_context, spheres  # noqa: E402

import paper_1506_03745_gb300 as pgb  # noqa: E402


def _solve(ctx, mode, tol=1e-8):
    x = torch.empty(pgb.pgb_num_unknowns(ctx), dtype=torch.float64, device="cuda")
    code, st = pgb.pgb_solve(ctx, mode, tol, 500, 100, x)
    assert code == 0, st
    return x


def _near(ctx):
    return pgb.pgb_keep_limit(ctx)["near"]


def test_a_refinement_stores_the_near_field_it_iterates_with():
    """Not another one for the FP64 products of its outer residual."""
    held = {}
    for residual in (0, 1):
        ctx = gpu_context(spheres(level_mol=3, level_srf=2), residual=residual)
        try:
            _solve(ctx, pgb.PGB_FP32_REFINE)
            held[residual] = _near(ctx)
        finally:
            pgb.pgb_destroy(ctx)
    assert held[0] == held[1] > 0
