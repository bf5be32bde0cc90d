"""Where lb_diagnostics leaves its result: behind the staged positions of a
context with cells, in a piece of its own before the first step and without
cells.  Position readbacks and diagnostics in turn disturb neither."""
import numpy as np
import pytest

from paper_1110_0995_gb300 import lbibm, scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def test_diagnostics_and_readbacks_in_turn():
    sc = scene.small_filter(seed=5, steps=0)
    n = int(np.prod(sc.dims))

    def run(before):
        sim = lbibm.Simulation.from_scene(sc)
        sim.set_deterministic(True)
        fluid = n - int(sim.solid_mask().sum())
        if before:
            d = sim.diagnostics()
            assert d[0] == pytest.approx(fluid, rel=1e-12) and not np.any(d[1:5])
        out = []
        for _ in range(3):
            sim.step(7)
            x = [sim.nodes(k) for k in range(len(sc.meshes))]
            d = np.array(sim.diagnostics())
            assert all(np.array_equal(sim.nodes(k), a) for k, a in enumerate(x))
            assert np.array_equal(d, sim.diagnostics()) and d[0] == pytest.approx(fluid, rel=1e-6) and d[5] > 0
            out.append((d, np.concatenate(x)))
        return out

    for (d, x), (e, y) in zip(run(False), run(True)):
        assert np.array_equal(d, e) and np.array_equal(x, y)


def test_without_cells():
    for _ in range(3):
        sim = lbibm.Simulation([lbibm.make_params((20, 12, 10), body_force=(1e-5, 0, 0))])
        a = sim.diagnostics()
        sim.step(5)
        b = sim.diagnostics()
        assert a[0] == pytest.approx(2400.0) and b[0] == pytest.approx(2400.0, rel=1e-6) and b[1] > a[1]
        sim.close()
