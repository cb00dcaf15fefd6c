"""GPU: what a context forms once, the near field of a solve's lists and the
panel moments of a geometry, is an interval of its own in the stage times."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from problems import gpu_context, spheres  # noqa: E402

import paper_1506_03745_gb300 as pgb  # noqa: E402


def _calls(ctx, run):
    pgb.pgb_timing(ctx, True, read=True)
    run()
    t = pgb.pgb_timing(ctx, False, read=True)
    assert all(ms >= 0 for ms, _ in (t[k] for k in ("p2p", "upward", "p2p_fp64", "upward_fp64")))
    return {k: t[k][1] for k in ("p2p", "upward", "p2p_fp64", "upward_fp64")}


@pytest.mark.parametrize("mode,stage", [(pgb.PGB_FP32, "p2p"), (pgb.PGB_FP64, "p2p_fp64")])
def test_forming_the_near_field_is_in_the_p2p_stage(mode, stage):
    ctx = gpu_context(spheres(level_mol=2, level_srf=2), graphs=0)
    try:
        x = torch.empty(pgb.pgb_num_unknowns(ctx), dtype=torch.float64, device="cuda")
        first, second = (_calls(ctx, lambda: pgb.pgb_solve(ctx, mode, 1e-5, 200, 100, x)) for _ in range(2))
        assert first[stage] == second[stage] + 1
    finally:
        pgb.pgb_destroy(ctx)


@pytest.mark.parametrize("precision,stage", [(pgb.PGB_FP32, "upward"), (pgb.PGB_FP64, "upward_fp64"), (pgb.PGB_FP64_DS, "upward_fp64")])
def test_forming_the_panel_moments_is_in_the_upward_stage(precision, stage):
    ctx = gpu_context(spheres(level_mol=2, level_srf=2), graphs=0)
    try:
        x = torch.tensor(np.random.default_rng(1).normal(size=pgb.pgb_num_unknowns(ctx)), device="cuda",
                         dtype=torch.float32 if precision == pgb.PGB_FP32 else torch.float64)
        y = torch.empty_like(x)
        first, second = (_calls(ctx, lambda: pgb.pgb_matvec(ctx, x, y, precision)) for _ in range(2))
        assert (first[stage], second[stage]) == (2, 1)
    finally:
        pgb.pgb_destroy(ctx)
