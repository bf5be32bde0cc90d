"""The FP32 stream-collide's wide form (one channel, 8192 blocks of 128 nodes
and more) against the oracle: the smallest lattices that take it, with rows
that are whole blocks and rows that break inside warps, and the lattice one
block short of it."""
import numpy as np
import pytest

import oracle
from paper_1110_0995_gb300 import scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("dims", [(256, 64, 64), (257, 64, 64), (128, 8191, 1)])
def test_wide_form_matches_the_oracle(dims):
    from paper_1110_0995_gb300 import lbibm

    sph = np.array([[9.0, 11.5, 8.25, 3.0], [100.5, 30.0, 12.0, 2.5], [120.0, 17.0, 0.0, 2.0]], np.float32)
    sc = scene.Scene("wide", dims, tau=0.8, body_force=(2e-5, -1e-5, 5e-6), periodic=(1, 0, 1),
                     wall_velocity=((0.02, 0, 0.01), (0, 0, 0)), spheres=sph)
    sim, ref = lbibm.Simulation.from_scene(sc), oracle.System.from_scene(sc)
    f0 = ref.get_f() * (1 + 0.01 * scene.random_field(7, (19, ref.N)))
    f0[:, ref.solid == 1] = ref.get_f()[:, ref.solid == 1]
    ref.set_f(f0)
    sim.set_populations(f0)
    sim.step(3)
    ref.step(3)
    fluid = ref.solid == 0
    # FP32 populations of size <= 1/3 and three collisions: as the other variants' parity tests
    np.testing.assert_allclose(sim.populations()[:, fluid], ref.get_f()[:, fluid], rtol=0, atol=2e-7)
