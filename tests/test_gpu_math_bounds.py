"""GPU: the FP64 1/sqrt and 2^x of the panel sums at the accuracy that they
claim, over their whole range and where their reductions break."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1506_03745_gb300 as pgb  # noqa: E402


def test_exp2_between_its_table_entries_and_at_their_edges():
    """Truncation (ln 2 / 64)^6 / 6! = 2.3e-15, the series' and the table's rounding
    and their product's 2^-52 each: 4e-15 with NumPy's own."""
    rng = np.random.default_rng(21)
    n = np.arange(-32 * 1019, 32 * 1000, 7)
    edges = n / 32.0 + 1.0 / 64.0
    t = np.concatenate([rng.uniform(-1019, 1000, 100000), rng.uniform(-1, 1, 50000), edges, np.nextafter(edges, np.inf),
                        np.nextafter(edges, -np.inf), n / 32.0])
    out = pgb.pgb_math_check(t)[:, 2]
    assert np.abs(out / np.exp2(t) - 1).max() <= 4e-15


def test_exp2_at_its_cut_off():
    """Below -1020 a value is zero or right; zero from the upper word after
    -1020's on, 2^-11 below."""
    t = -1020.0 - np.concatenate([np.linspace(0.0, 1.0, 4097)[1:], 2.0 ** -np.arange(12.0, 42.0)])
    out = pgb.pgb_math_check(t)[:, 2]
    right = np.abs(out / np.exp2(t) - 1) <= 4e-15
    assert np.all(right | (out == 0.0))
    assert np.all(out[t <= -1020.0 - 2.0 ** -11] == 0.0)
    assert pgb.pgb_math_check(np.array([-1020.0]))[0, 2] == 2.0 ** -1020


def test_rsqrt_over_the_double_range():
    """One Halley step from an estimate good to 2^-20 leaves (5/2) 2^-60; the
    rest is the rounding of its last three operations."""
    rng = np.random.default_rng(22)
    x = np.concatenate([10.0 ** rng.uniform(-290, 290, 200000), 4.0 ** np.arange(-480, 481, 3.0)])
    out = pgb.pgb_math_check(x)
    ref = 1.0 / np.sqrt(x.astype(np.longdouble))
    assert float(np.abs(out[:, 1].astype(np.longdouble) / ref - 1).max()) <= 3 * 2.0 ** -53
    assert np.array_equal(out[:, 0], out[:, 1])
