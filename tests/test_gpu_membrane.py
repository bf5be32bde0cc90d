"""The patch-wise membrane kernel against the oracle's forces: meshes of one
small patch up to many, a hub node of the largest valence, triangulations with
mixed valences, cells much larger than the lattice spacing (coarser position
grid), several connectivities in one context, a cell far from where it rested."""
import numpy as np
import pytest

import oracle
from paper_1110_0995_gb300 import scene

pytestmark = pytest.mark.gpu

MODULI = (0.01, 0.01, 0.01, 0.5, 0.9)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _tetra():
    v = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1.0]])
    return v, np.array([[0, 1, 2], [0, 3, 1], [0, 2, 3], [1, 3, 2]], np.int32)


def _bipyramid(k):
    a = 2 * np.pi * np.arange(k) / k
    v = np.vstack([np.c_[np.cos(a), np.sin(a), 0 * a], [[0, 0, 1], [0, 0, -1.0]]])
    t = [(i, (i + 1) % k, k) for i in range(k)] + [((i + 1) % k, i, k + 1) for i in range(k)]
    return v, np.array(t, np.int32)


MESHES = {"tetra": _tetra, "ico0": lambda: scene.icosphere(0), "ico1": lambda: scene.icosphere(1),
          "ico2": lambda: scene.icosphere(2), "fib107": lambda: scene.fibonacci_sphere_mesh(107),
          "fib108": lambda: scene.fibonacci_sphere_mesh(108), "fib109": lambda: scene.fibonacci_sphere_mesh(109),
          "fib217": lambda: scene.fibonacci_sphere_mesh(217), "hub64": lambda: _bipyramid(64),
          "rbc": lambda: scene.cell_template("rbc"), "ico5": lambda: scene.icosphere(5)}


def _placed(name, radius, centre, seed):
    if name.startswith("fib"):
        pytest.importorskip("scipy")
    v, t = MESHES[name]()
    rng = np.random.default_rng(seed)
    rest = scene.quantize(radius * v @ scene.random_rotation(rng).T + centre, scene.POS_QUANTUM)
    edge = np.linalg.norm(rest[t[:, 0]] - rest[t[:, 1]], axis=1).mean()
    now = scene.quantize(rest * [1.01, 0.99, 1.02] + 0.01 * edge * rng.standard_normal(rest.shape), scene.POS_QUANTUM)
    return rest, np.ascontiguousarray(t, np.int32), now


def _check(sim, k, rest, tris, now):
    ref = oracle.mesh_forces(now, rest, tris, MODULI)
    # FP32 element geometry: the repository's bound for node forces, 1e-5 of the largest
    assert np.abs(sim.forces(k) - ref).max() <= 1e-5 * np.abs(ref).max()


@pytest.mark.parametrize("name,radius", [(n, 6.0) for n in MESHES] + [("ico2", 0.6), ("ico2", 150.0), ("rbc", 60.0)])
def test_forces_of_one_mesh(name, radius):
    from paper_1110_0995_gb300 import lbibm

    rest, tris, now = _placed(name, radius, np.array([20.0, 18.0, 16.0]), 3)
    sim = lbibm.Simulation([lbibm.make_params((40, 36, 32), periodic=(1, 1, 1))])
    sim.add_mesh(rest, tris, MODULI)
    sim.set_nodes(0, now)
    sim.step(1)
    _check(sim, 0, rest, tris, now)


def test_forces_of_mixed_meshes_far_from_rest():
    from paper_1110_0995_gb300 import lbibm

    sim = lbibm.Simulation([lbibm.make_params((64, 48, 40), periodic=(1, 1, 1))])
    placed = []
    for k, (name, radius) in enumerate([("rbc", 1.0), ("ico2", 5.0), ("tetra", 2.0), ("rbc", 1.1), ("hub64", 4.0),
                                        ("ico1", 3.0), ("ico2", 6.0)]):
        rest, tris, now = _placed(name, radius, np.array([8.0 + 7 * k, 20.0, 18.0]), k)
        if k in (1, 3):                       # carried along the channel, several periods
            now = now + np.array([640.0, 0.0, 0.0])
        placed.append((rest, tris, now))
        sim.add_mesh(rest, tris, MODULI)
        sim.set_nodes(k, now)
    sim.step(1)
    for k, p in enumerate(placed):
        _check(sim, k, *p)
