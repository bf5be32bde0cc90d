"""lb_diagnostics against FP64 sums of the same populations on the host: one
node to several blocks, obstacles, ordinary flow, a state at rest, tiny and
large moments (the FP64 path), non-finite populations."""
import numpy as np
import pytest

import oracle
from paper_1110_0995_gb300 import scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _sim(dims, storage="f32", spheres=()):
    from paper_1110_0995_gb300 import lbibm

    sph = np.array(spheres, np.float32).reshape(-1, 4)
    return lbibm.Simulation.from_scene(scene.Scene("d", dims, tau=0.9, body_force=(1e-4, -2e-5, 3e-5), periodic=(1, 1, 1),
                                                   spheres=sph), storage)


def _expected(sim, G=(1e-4, -2e-5, 3e-5)):
    """Mass, momentum and largest speed in FP64 from rho, u of the last collision."""
    rho, u = (a.astype(np.float64) for a in sim.fields())
    fluid = sim.solid_mask() == 0
    G = np.array(G)[:, None]
    mom = (rho * u + 0.5 * G)[:, fluid]
    return rho[fluid].sum(), mom.sum(1), np.sqrt((u[:, fluid] ** 2).sum(0)).max(), np.abs(mom).sum(1)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("dims,spheres", [((1, 1, 1), ()), ((5, 3, 7), ()), ((36, 23, 19), ((9.0, 11.5, 8.25, 3.0),)),
                                          ((128, 96, 64), ((60.0, 40.0, 30.0, 9.0),))])
def test_sums_and_largest_speed(dims, spheres, storage):
    sim = _sim(dims, storage, spheres)
    w = oracle.constants()[1]
    f = w[:, None] * (1 + 0.02 * scene.random_field(3, (19, sim.N)))
    sim.set_populations(f)
    sim.step(3)
    mass, mom, speed, size = _expected(sim)
    d = sim.diagnostics()
    # the fields are FP32 (rounded once per node): half an ulp of every term
    assert abs(d[0] - mass) <= 2.0 ** -24 * mass
    assert (np.abs(d[1:4] - mom) <= 2.0 ** -22 * size + 1e-12).all()
    assert abs(d[5] - speed) <= 4 * 2.0 ** -24 * speed
    assert d[4] == 0


def test_rest_uniform_and_extreme_states():
    sim = _sim((24, 8, 8))
    assert np.array_equal(sim.diagnostics(), [sim.N, 0, 0, 0, 0, 0])   # before any step
    w = oracle.constants()[1]
    e1 = np.zeros(19)
    e1[1], e1[2] = 1.0, -1.0
    for scale, drho in ((0.0, 0.0), (1e-14, 0.0), (3e-3, 0.0), (0.9, 0.5), (40.0, 90.0)):
        sim = _sim((24, 8, 8))
        f = np.repeat((w * (1 + drho) + scale / 2 * e1)[:, None], sim.N, axis=1)
        f[1, 7] += 1e-3 * scale                       # one node a little faster
        sim.set_populations(f)
        sim.step(1)
        mass, mom, speed, size = _expected(sim)
        d = sim.diagnostics()
        assert abs(d[0] - mass) <= 2.0 ** -23 * mass
        assert (np.abs(d[1:4] - mom) <= 2.0 ** -21 * (size + mass)).all()
        # u is formed from momenta of FP32 populations whose size is the density's deviation
        assert abs(d[5] - speed) <= 8 * 2.0 ** -24 * (speed + drho)


def test_non_finite_populations_are_counted():
    import ctypes

    sim = _sim((24, 8, 8))
    sim.step(2)
    state = bytearray(sim.save_state())
    # the first populations of direction 0 follow the header; three of them become NaN / inf
    head = 40
    assert ctypes.sizeof(ctypes.c_double) == 8
    for k, v in ((3, np.nan), (4, np.inf), (700, -np.inf)):
        state[head + 4 * k:head + 4 * k + 4] = np.float32(v).tobytes()
    sim.load_state(bytes(state))
    d = sim.diagnostics()
    assert d[4] == 3
    assert np.isinf(d[5])
    assert not np.isfinite(d[0])
