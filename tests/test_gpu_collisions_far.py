"""Collision forces more than 2048 lu from the origin, where one 32-bit part of
a fixed-point coordinate no longer holds it: cells carried that far along a
periodic channel whose period is no power of two (contacts between cells, with
a bead, and none), and the walls of an axis longer than that."""
import numpy as np
import pytest

import oracle
from paper_1110_0995_gb300 import lbibm, scene

pytestmark = pytest.mark.gpu

ZERO = (0.0,) * 5


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _compare(sc, moved):
    sim, ref = lbibm.Simulation.from_scene(sc), oracle.System.from_scene(sc)
    for k, x in moved.items():
        sim.set_nodes(k, x)
        ref.set_nodes(k, x)
    sim.step(1)
    ref.step(1)
    F = [sim.forces(k) for k in range(len(sc.meshes))]
    Fo = [ref.forces(k) for k in range(len(sc.meshes))]
    big = max(np.abs(f).max() for f in Fo)
    assert big > 1e-3
    for f, fo in zip(F, Fo):
        assert np.abs(f - fo).max() < 1e-5 * big        # the repository's bound for collision forces
    assert sim.diagnostics()[4] == 0
    return Fo


def _sphere(radius, centre):
    v, t = scene.icosphere(2)
    return scene.Mesh("x", scene.quantize(radius * v + centre, scene.POS_QUANTUM), np.ascontiguousarray(t, np.int32), ZERO)


@pytest.mark.parametrize("periods", [(22, 22, 22, 22), (22, 0, -30, 0), (0, -22, 0, 43), (-1000, 30000, 0, 22)])
def test_cells_far_down_a_periodic_channel(periods):
    dims = (96, 40, 36)
    # two cells in contact, a third touching a bead, a fourth across the box's edge from the first
    meshes = [_sphere(4.0, [4.2, 18.0, 17.0]), _sphere(4.0, [12.4, 19.0, 17.0]), _sphere(4.0, [60.0, 20.0, 18.0]),
              _sphere(4.0, [92.1, 17.5, 17.0])]
    sc = scene.Scene("far", dims, periodic=(1, 0, 0), spheres=np.array([[66.3, 20.5, 18.0, 2.0]], np.float32),
                     repulsion=(0.01, 1.0), meshes=meshes)
    Fo = _compare(sc, {k: m.rest + [n * dims[0], 0.0, 0.0] for k, (m, n) in enumerate(zip(meshes, periods))})
    assert all(np.abs(f).max() > 1e-4 for f in Fo)


def test_walls_of_a_long_axis():
    dims = (20, 2500, 20)
    meshes = [_sphere(4.0, [10.0, 4.0, 9.0]), _sphere(4.0, [10.0, 1200.0, 10.0]), _sphere(4.0, [9.0, 2300.0, 10.0]),
              _sphere(4.0, [10.0, 2495.2, 10.0])]
    sc = scene.Scene("walls", dims, periodic=(1, 0, 0), repulsion=(0.01, 1.0), meshes=meshes)
    Fo = _compare(sc, {})
    assert np.abs(Fo[0]).max() > 1e-4 and np.abs(Fo[3]).max() > 1e-4
    assert np.abs(Fo[1]).max() == 0.0 and np.abs(Fo[2]).max() == 0.0
