"""GPU: the charge weights and reaction potentials by the far rule's orbits, for
every far rule, few and many charges, some within the close-by rule's reach,
against the oracle's energies of the same vector."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.energy import energies  # noqa: E402
from problems import gpu_context, oracle_system, spheres  # noqa: E402

import paper_1506_03745_gb300 as pgb  # noqa: E402


@pytest.mark.parametrize("K", [1, 3, 4, 7])
@pytest.mark.parametrize("nq", [3, 31, 32, 77])
def test_energies_match_the_oracle(K, nq):
    """A term is good to 1e-14 (the squared distance loses a factor |d|^2 / r^2
    below ten) and the two kinds of term cancel by less than 1e3."""
    bodies = spheres(level_srf=1, kind="sigma", mol_nu=4)
    rng = np.random.default_rng(nq)
    u = rng.normal(size=(nq, 3))
    u *= (rng.uniform(0.1, 3.3, nq) / np.linalg.norm(u, axis=1))[:, None]
    bodies[0].update(qxyz=u, q=rng.uniform(0.2, 1.0, nq))
    system = oracle_system(bodies, theta=0.0, K=K)
    x = rng.uniform(0.5, 1.5, system.n)
    ref = energies(system, x)
    ctx = gpu_context(bodies, theta=0.0, K=K)
    try:
        xd = torch.tensor(x, device="cuda")
        for got in (pgb.pgb_energy(ctx, xd), pgb.pgb_energy_noalloc(ctx, xd)):
            assert got["solvation"] == pytest.approx(ref["solvation"], rel=1e-10)
            assert got["coulomb"] == pytest.approx(ref["coulomb"], rel=1e-10)
    finally:
        pgb.pgb_destroy(ctx)
