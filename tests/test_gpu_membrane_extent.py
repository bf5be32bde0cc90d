"""Membrane forces of cells that reach further from their reference node than
the position grid holds in 24 or 32 bits: a cell pulled out by its reference
node, so that all others are far from it (their own elements still of ordinary
size), and a mesh tens of thousands of lattice units across."""
import numpy as np
import pytest

import oracle
from paper_1110_0995_gb300 import lbibm, scene

pytestmark = pytest.mark.gpu

LOCAL = (0.01, 0.01, 0.01, 0.0, 0.0)      # stretching, bending, local area


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


def _forces(rest, tris, now):
    sim = lbibm.Simulation([lbibm.make_params((40, 36, 32), periodic=(1, 1, 1))])
    sim.add_mesh(rest, tris, LOCAL)
    sim.set_nodes(0, now)
    sim.step(1)
    return sim.forces(0)


def _perturbed(rest, tris, seed):
    edge = np.linalg.norm(rest[tris[:, 0]] - rest[tris[:, 1]], axis=1).mean()
    return scene.quantize(rest * [1.01, 0.99, 1.02] + 0.01 * edge * np.random.default_rng(seed).standard_normal(rest.shape),
                          scene.POS_QUANTUM)


def _check_far(F, ref, tris):
    # nodes whose elements (triangles and their neighbours over an edge) do not touch node 0
    near = {0}
    for _ in range(2):
        near |= set(tris[np.isin(tris, list(near)).any(1)].ravel().tolist())
    far = np.setdiff1d(np.arange(len(F)), list(near))
    assert len(far) > 600
    # FP32 element geometry: the repository's bound for node forces, 1e-5 of the largest
    assert np.abs(F[far] - ref[far]).max() <= 1e-5 * np.abs(ref[far]).max()


@pytest.mark.parametrize("shift", [100.0, 300.0, 3000.0, 40000.0, -1.0e6])
def test_nodes_far_from_the_reference_node(shift):
    v, t = scene.icosphere(3)
    rest, tris = scene.quantize(6.0 * v + [20.0, 18.0, 16.0], scene.POS_QUANTUM), np.ascontiguousarray(t, np.int32)
    now = _perturbed(rest, tris, 1)
    now[1:] += [shift, 0.25 * shift, -0.5 * shift]
    F, ref = _forces(rest, tris, now), oracle.mesh_forces(now, rest, tris, LOCAL)
    _check_far(F, ref, tris)


def test_among_many_cells():
    """Enough patches for the kernel's form of four blocks per SM."""
    v, t = scene.icosphere(3)
    tris = np.ascontiguousarray(t, np.int32)
    sim = lbibm.Simulation([lbibm.make_params((40, 36, 32), periodic=(1, 1, 1))])
    cells = []
    for k in range(80):
        rest = scene.quantize(6.0 * v + [20.0 + 0.25 * k, 18.0, 16.0], scene.POS_QUANTUM)
        now = _perturbed(rest, tris, k)
        if k in (0, 41, 79):
            now[1:] += [3000.0, 40000.0, -70.0]
        sim.add_mesh(rest, tris, LOCAL)
        sim.set_nodes(k, now)
        cells.append((rest, now))
    sim.step(1)
    for k, (rest, now) in enumerate(cells):
        F, ref = sim.forces(k), oracle.mesh_forces(now, rest, tris, LOCAL)
        if k in (0, 41, 79):
            _check_far(F, ref, tris)
        else:
            assert np.abs(F - ref).max() <= 1e-5 * np.abs(ref).max()


@pytest.mark.parametrize("radius", [60.0, 6000.0, 20000.0, 500000.0])
def test_meshes_of_large_extent(radius):
    v, t = scene.icosphere(3)
    rest, tris = scene.quantize(radius * v + [20.0, 18.0, 16.0], scene.POS_QUANTUM), np.ascontiguousarray(t, np.int32)
    now = _perturbed(rest, tris, 2)
    F, ref = _forces(rest, tris, now), oracle.mesh_forces(now, rest, tris, LOCAL)
    assert np.abs(F - ref).max() <= 1e-5 * np.abs(ref).max()
