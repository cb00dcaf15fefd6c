"""GPU: a caller's stream capture of a product that is the first on its
geometry (graphs = 0: a captured stream takes no graph launches).  What the
capture records has not run yet: products made before the first replay, and
after it, are those of the new geometry."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from problems import gpu_context, star_molecule  # noqa: E402

import paper_1506_03745_gb300 as pgb  # noqa: E402


@pytest.mark.parametrize("precision", [pgb.PGB_FP32, pgb.PGB_FP64, pgb.PGB_FP64_DS])
def test_products_around_a_captured_first_product(precision):
    c, s = np.cos(1.0), np.sin(1.0)
    R = np.array([[c, -s, 0.0], [s, c, 0.0], [0.0, 0.0, 1.0]])
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = gpu_context(star_molecule(nu=8), graphs=0, leaf_size=8)
        try:
            dtype = torch.float32 if precision == pgb.PGB_FP32 else torch.float64
            x = torch.tensor(np.random.default_rng(3).normal(size=pgb.pgb_num_unknowns(ctx)), device="cuda", dtype=dtype)
            want, got, held = torch.empty_like(x), torch.empty_like(x), torch.zeros_like(x)
            pgb.pgb_set_pose(ctx, 0, R, np.zeros(3))
            pgb.pgb_tree_build(ctx)
            pgb.pgb_matvec(ctx, x, want, precision)
            pgb.pgb_set_pose(ctx, 0, np.eye(3), np.zeros(3))  # another geometry, and its products
            pgb.pgb_tree_build(ctx)
            pgb.pgb_matvec(ctx, x, got, precision)
            pgb.pgb_set_pose(ctx, 0, R, np.zeros(3))
            pgb.pgb_tree_build(ctx)
            graph = torch.cuda.CUDAGraph()
            stream.synchronize()
            with torch.cuda.graph(graph, stream=stream):
                pgb.pgb_matvec(ctx, x, held, precision)
            # the moments of one geometry, formed beforehand or on the spot: a few hundred roundings
            tol = 200 * {pgb.PGB_FP32: 2.0 ** -24, pgb.PGB_FP64: 2.0 ** -53, pgb.PGB_FP64_DS: 2.0 ** -47}[precision]
            for y in (got, held, got):
                y.zero_()
                if y is held:
                    graph.replay()
                else:
                    pgb.pgb_matvec(ctx, x, y, precision)
                stream.synchronize()
                assert float(torch.linalg.norm(y - want)) <= tol * float(torch.linalg.norm(want))
        finally:
            stream.synchronize()
            pgb.pgb_destroy(ctx)
