"""The 16-bit four-node stream-collide in its three forms (one channel, several
channels, a moving wall somewhere): a channel's populations do not depend on
which form advanced it.  The forms share their arithmetic and their rounding
is a function of the channel's own node indices and moments, so a batch whose
first channel equals a single context agrees with it bit for bit; the other
channels (whose node indices are shifted by the batch) agree with the oracle
within the 16-bit rounding of one step."""
import numpy as np
import pytest

import oracle
from paper_1110_0995_gb300 import scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _scene(dims, wall, seed):
    rng = np.random.default_rng(seed)
    sph = scene.quantize(np.column_stack([rng.uniform(0, dims[0], 3), rng.uniform(0, dims[1], 3),
                                          rng.uniform(0, dims[2], 3), rng.uniform(0.6, 1.6, 3)]),
                         scene.SPHERE_QUANTUM).astype(np.float32)
    return scene.Scene("quad", dims, tau=0.8, body_force=(2e-4, -1e-4, 5e-5), periodic=(1, 0, 1),
                       wall_velocity=(((0.02, 0, 0.01) if wall else (0, 0, 0)), (0, 0, 0)), spheres=sph)


# rows that break inside a warp, one row per block piece, a padded last quad
@pytest.mark.parametrize("dims", [(4, 4, 4), (36, 7, 5), (256, 5, 3), (512, 4, 4)])
@pytest.mark.parametrize("walls", [(False, False), (True, False), (False, True)])
@pytest.mark.parametrize("storage", ["f16", "bf16"])
def test_batch_channel_equals_single_context(dims, walls, storage):
    from paper_1110_0995_gb300 import lbibm

    a, b = _scene(dims, walls[0], 1), _scene((20, 6, 7), walls[1], 2)
    batch, alone = lbibm.Simulation.from_scenes([a, b], storage), lbibm.Simulation.from_scene(a, storage)
    refs = [oracle.System.from_scene(s) for s in (a, b)]
    for ch, ref in enumerate(refs):
        f = ref.get_f() * (1 + 0.01 * scene.random_field(5 + ch, (19, ref.N)))
        f[:, ref.solid == 1] = ref.get_f()[:, ref.solid == 1]
        batch.select(ch)
        batch.set_populations(f)
        start = batch.populations()               # (as the 16-bit storage holds them)
        if ch == 0:
            alone.set_populations(f)
        ref.set_f(start)
    for sim in (batch, alone):
        assert sim.kernel_config() == (4, 64)
        sim.step(1)
    batch.select(0)
    assert np.array_equal(batch.populations(), alone.populations())
    # one stochastic rounding of each stored value h_i / w_i: below one unit in
    # the last place (2^-10, 2^-7 of the value), plus the FP32 collision's error
    ulp = {"f16": 2.0 ** -10, "bf16": 2.0 ** -7}[storage]
    _, w, _ = oracle.constants()
    for ch, ref in enumerate(refs):
        ref.step(1)
        batch.select(ch)
        fluid = ref.solid == 0
        h = ref.get_f()[:, fluid] - w[:, None]
        err = np.abs(batch.populations()[:, fluid] - w[:, None] - h)
        assert (err <= ulp * np.abs(h) + 2e-7 * w[:, None]).all()
    # and further steps in all forms
    for sim in (batch, alone):
        sim.step(7)
    batch.select(0)
    assert np.array_equal(batch.populations(), alone.populations())
