"""Collision forces between cells against the oracle where the node-node kernel
cuts its work: cells of one unit of 128 nodes and one node more, cells of
several tiles, partners in all directions, across the periodic boundary, a
cell many periods down the channel, and one out of reach."""
import numpy as np
import pytest

import oracle
from paper_1110_0995_gb300 import scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _mesh(kind):
    if kind.startswith("fib"):
        pytest.importorskip("scipy")
        v, t = scene.fibonacci_sphere_mesh(int(kind[3:]))
        return 2.0 * v, t
    return scene.cell_template(kind)


@pytest.mark.parametrize("periodic", [(1, 0, 0), (1, 1, 1), (0, 0, 0)])
@pytest.mark.parametrize("a,b,gap", [("fib128", "fib129", 0.3), ("rbc", "rbc", 0.2), ("ctc", "rbc", 0.4),
                                     ("ctc", "ctc", 0.5), ("fib513", "fib127", -0.5)])
def test_node_forces_match_the_oracle(a, b, gap, periodic):
    from paper_1110_0995_gb300 import lbibm

    dims, zero = (64, 48, 40), (0.0,) * 5
    rng = np.random.default_rng(5)
    (va, ta), (vb, tb) = _mesh(a), _mesh(b)
    ra, rb = (np.linalg.norm(v, axis=1).max() for v in (va, vb))
    meshes, shift = [], []
    first = va @ scene.random_rotation(rng).T
    centre = np.array([20.0, 22.0, 18.0])
    meshes.append((first + centre, ta))
    for d in ([1.0, 0.2, 0.1], [-0.3, 1.0, 0.4], [0.1, -0.5, -1.0]):    # partners around the first cell
        d = np.array(d) / np.linalg.norm(d)
        v = vb @ scene.random_rotation(rng).T
        # surfaces `gap` apart along d
        reach = (first @ d).max() + (-(v @ d)).max() + gap
        meshes.append((v + centre + d * reach, tb))
    meshes.append((vb + [62.5, 8.0, 8.0] if periodic[0] else vb + [50.0, 8.0, 8.0], tb))
    meshes.append((vb + [62.5 + 2 * rb + 0.4, 8.0, 8.2] if periodic[0] else vb + [50.0, 8.0 + 2 * rb + 0.4, 8.2], tb))
    spheres = np.array([[40.0, 40.0, 30.0, 2.0]], np.float32)
    sc = scene.Scene("units", dims, periodic=periodic, spheres=spheres, repulsion=(0.01, 1.0),
                     meshes=[scene.Mesh("x", scene.quantize(v, scene.POS_QUANTUM), np.ascontiguousarray(t, np.int32), zero)
                             for v, t in meshes])
    sim, ref = lbibm.Simulation.from_scene(sc), oracle.System.from_scene(sc)
    if periodic[0]:                                     # the first partner three periods on
        moved = sc.meshes[1].rest + [3 * dims[0], 0.0, 0.0]
        sim.set_nodes(1, moved)
        ref.set_nodes(1, moved)
    sim.step(1)
    ref.step(1)
    F = np.concatenate([sim.forces(k) for k in range(len(meshes))])
    Fo = np.concatenate([ref.forces(k) for k in range(len(meshes))])
    assert np.abs(Fo).max() > 1e-3
    assert np.abs(F - Fo).max() < 1e-5 * np.abs(Fo).max()      # the repository's bound for collision forces
    assert sim.diagnostics()[4] == 0
