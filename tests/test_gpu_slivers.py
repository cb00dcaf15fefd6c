"""GPU: P2P sums of a long thin panel at targets close to its quadrature points
and far from its centroid.

A triangle 10 long and 0.05 high, with small triangles as targets 0.01 above
those points of the far rule that lie outside the close-by distance.  FP32:
target, centroid, their difference, the point's offset from the centroid and
the sum of both round at 2^-24 of at most 5 each, within 16 * 2^-24 a component
or 1.7e-6 in all, which is 1.7e-4 of the distance 0.01; 1/r takes that once, the
double layer's n.(x - y) / r^3 four times: 7e-4.  A squared distance formed as a
difference of terms of up to 12 would be off by 1e-6 or more of 1e-4.  FP64:
2^-53 for 2^-24 makes 1.3e-12, and the reference's points (1e-15 of 10, over
0.01, four times) as much again: 3e-12."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.quadrature import triangle_rule  # noqa: E402
from problems import gpu_context  # noqa: E402

import paper_1506_03745_gb300 as pgb  # noqa: E402

HEIGHT, KAPPA = 0.01, 0.125


def _bodies(K):
    needle = np.array([[0.0, 0.0, 0.0], [10.0, 0.0, 0.0], [5.0, 0.05, 0.0]])
    mu, w = triangle_rule(K)
    y = (mu + 1.0 / 3.0) @ needle
    area = 0.5 * 10.0 * 0.05
    at = y[((y - needle.mean(0)) ** 2).sum(1) > 8.0 * area * 1.1] + [0.0, 0.0, HEIGHT]
    small = 1e-3 * np.array([[1.0, 0.0, 0.0], [-0.5, 0.8, 0.0], [-0.5, -0.8, 0.0]])
    verts = np.concatenate([needle] + [a + small for a in at])
    tris = np.arange(len(verts), dtype=np.int32).reshape(-1, 3)
    body = dict(kind="dielectric", verts=verts, tris=tris, eps_in=4.0, qxyz=np.zeros((1, 3)), q=np.array([1.0]), bc=0.0)
    return [body], verts[tris[1:]].mean(1), y, np.asarray(w) * area


@pytest.mark.parametrize("precision,tol", [("fp32", 7e-4), ("fp64", 3e-12)])
@pytest.mark.parametrize("K", [3, 4, 7])
def test_targets_over_the_points_of_a_needle(K, precision, tol):
    bodies, at, y, w = _bodies(K)
    assert len(at) >= 2
    n = len(at) + 1
    d = at[:, None] - y[None]
    r = np.sqrt((d * d).sum(-1))
    nd = d[..., 2]
    e, inv = np.exp(-KAPPA * r), 1.0 / (4.0 * np.pi)
    V = inv * (w / r).sum(1), inv * (w * e / r).sum(1)
    D = inv * (w * nd / r ** 3).sum(1), inv * (w * nd * e * (1 + KAPPA * r) / r ** 3).sum(1)
    ctx = gpu_context(bodies, kappa=KAPPA, theta=0.0, K=K)
    try:
        for layer in (0, 1):  # phi or its normal derivative on the needle alone
            x = np.zeros(2 * n)
            x[layer * n] = 1.0
            xt = torch.tensor(x, device="cuda", dtype=torch.float32 if precision == "fp32" else torch.float64)
            out = torch.empty_like(xt)
            pgb.pgb_matvec(ctx, xt, out, pgb.PGB_FP32 if precision == "fp32" else pgb.PGB_FP64)
            out = out.double().cpu().numpy()
            want = (D[0], -D[1]) if layer == 0 else (-V[0], 4.0 / 80.0 * V[1])
            for rows, ref in ((out[1:n], want[0]), (out[n + 1:], want[1])):
                assert np.abs(rows / ref - 1.0).max() <= tol, (layer, rows / ref - 1.0)
    finally:
        pgb.pgb_destroy(ctx)
