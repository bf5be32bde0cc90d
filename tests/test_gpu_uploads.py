"""Steps right behind an upload: a loaded state and set populations are on the
device when the next lb_step starts, whatever the lattice's size (the copies
run on the context's stream).  Mesh-free contexts, so runs repeat bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _sim(dims, storage):
    from paper_1110_0995_gb300 import lbibm

    return lbibm.Simulation([lbibm.make_params(dims, body_force=(1e-5, 2e-6, 0.0), periodic=(1, 0, 0), storage=storage)])


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("dims", [(20, 9, 7), (256, 128, 64)])
def test_steps_behind_a_loaded_state(dims, storage):
    a = _sim(dims, storage)
    a.step(11)
    state = a.save_state()
    a.step(6)
    want = a.fields()[1]
    for _ in range(4):
        b = _sim(dims, storage)
        b.step(3)
        b.load_state(state)
        b.step(6)
        assert np.array_equal(b.fields()[1], want)
        b.close()


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("dims", [(20, 9, 7), (128, 64, 64)])
def test_steps_behind_set_populations(dims, storage):
    a = _sim(dims, storage)
    a.step(11)
    f = a.populations()
    a.set_populations(f)
    a.synchronize()
    a.step(6)
    want = a.fields()[1]
    for _ in range(3):
        b = _sim(dims, storage)
        b.step(11)
        b.set_populations(f)
        b.step(6)
        assert np.array_equal(b.fields()[1], want)
        b.close()
