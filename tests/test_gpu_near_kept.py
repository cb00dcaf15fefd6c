"""GPU: which near fields a context holds, and for how long (pgb_keep_limit
reports the bytes)."""
import numpy as np
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


@pytest.mark.parametrize("change", ["reset", "build", "refresh"])
def test_changed_lists_give_the_near_field_back(change):
    ctx = gpu_context(spheres(level_mol=3, level_srf=2))
    try:
        for mode in (pgb.PGB_FP32_REFINE, pgb.PGB_FP64):
            _solve(ctx, mode)
        first = _near(ctx)
        assert first > 0
        pgb.pgb_set_pose(ctx, 0, np.eye(3), np.array([-0.25, 0.0, 0.0]))
        {"reset": pgb.pgb_tree_reset, "build": pgb.pgb_tree_build, "refresh": pgb.pgb_tree_refresh}[change](ctx)
        assert _near(ctx) == 0
        if change == "reset":
            pgb.pgb_tree_build(ctx)
        x = _solve(ctx, pgb.PGB_FP32_REFINE)
        y, b = torch.empty_like(x), torch.empty_like(x)
        pgb.pgb_matvec(ctx, x, y, pgb.PGB_FP64)
        pgb.pgb_rhs(ctx, b)
        assert float(torch.linalg.norm(b - y) / torch.linalg.norm(b)) <= 2e-8
    finally:
        pgb.pgb_destroy(ctx)


@pytest.mark.parametrize("mode", [1, 2])
def test_a_large_near_field_goes_with_its_solve(mode):
    """More than a 32nd of its bound is given back at the end; the solutions of
    a solve that forms it anew and of one that may keep it are the same bits."""
    ctx = gpu_context(spheres(level_mol=3, level_srf=2))
    try:
        x = _solve(ctx, mode)
        size = _near(ctx)
        assert size > 0
        limit = max(pgb.pgb_keep_limit(ctx)["moments"], 2 * size)
        assert limit / 32 < size <= limit
        pgb.pgb_keep_limit(ctx, limit)
        pgb.pgb_tree_build(ctx)
        for _ in range(2):
            again = _solve(ctx, mode)
            assert pgb.pgb_keep_limit(ctx, limit)["near"] == 0
            assert torch.equal(x, again)
    finally:
        pgb.pgb_destroy(ctx)
