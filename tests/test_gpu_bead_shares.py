"""The bead kernel where it cuts its work: one tile and one bead more, odd
shares, shares of several stages, against the oracle; and two runs bit for bit."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _lattice(n, seed):
    """Beads on a jittered lattice (no two closer than 1.6), moments mostly along z."""
    rng = np.random.default_rng(seed)
    side = int(np.ceil(n ** (1 / 3)))
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)[:n]
    x = (g + 0.5) * 2.4 + rng.uniform(-0.4, 0.4, (n, 3))
    m = np.array([0.0, 0.0, 1.0]) + 0.2 * rng.standard_normal((n, 3))
    return x.astype(np.float32).astype(np.float64), m.astype(np.float32).astype(np.float64), side * 2.4


@pytest.mark.parametrize("periodic", [(0, 0, 0), (1, 1, 1), (0, 1, 0)])
@pytest.mark.parametrize("n", [2, 31, 128, 129, 1001, 9001])
def test_forces_match_the_oracle(n, periodic):
    from paper_1110_0995_gb300 import lbibm

    x, m, side = _lattice(n, n)
    args = (x, m, 0.5, 1.0, 5.0, (side,) * 3, periodic)
    F, Fo = lbibm.bead_forces(*args), oracle.bead_forces(*args)
    # the repository's bound for bead forces: 1e-5 of the largest
    assert np.abs(F - Fo).max() <= 1e-5 * np.abs(Fo).max()
    assert np.array_equal(F, lbibm.bead_forces(*args))


def test_relaxation_repeats_bit_for_bit():
    from paper_1110_0995_gb300 import lbibm

    x, m, side = _lattice(3001, 1)
    run = lambda: lbibm.bead_relax(x, m, 0.5, 1.0, 5.0, 0.2, 0.05, 12, (side,) * 3, (1, 1, 1))  # noqa: E731
    a = run()
    assert np.array_equal(a, run())
    assert np.abs(a - x).max() > 1e-3
