"""Points with mass: the membrane kernel of a cycle runs beside the
stream-collide of the one before it when the kernels are programmatic
dependents, and after it with ordinary launches.  The two schedules must agree
bit for bit in the deterministic cycle, with one and several cells, over whole
graphs of cycles and a remainder."""
import numpy as np
import pytest

from paper_1110_0995_gb300 import scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("dims,cells", [((57, 41, 23), (1, 0)), ((96, 48, 32), (4, 1)), ((192, 64, 48), (12, 2))])
def test_schedules_agree_bit_for_bit(dims, cells, storage):
    from paper_1110_0995_gb300 import lbibm

    sc = scene.small_filter(seed=9, dims=dims, n_rbc=cells[0], n_ctc=cells[1])
    sc.ib_dynamics = (2.0, 0.05)
    out = []
    for schedule in (0, 2):
        sim = lbibm.Simulation.from_scene(sc, storage)
        sim.set_deterministic(True)
        sim.set_schedule(schedule)
        for n in (1, 8, 19, 8):
            sim.step(n)
        rho, u = sim.fields()
        out.append([rho, u] + [f(m) for m in range(len(sc.meshes)) for f in (sim.nodes, sim.velocities)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    assert max(np.abs(v).max() for v in out[0][3::2]) > 0.0   # the points move
