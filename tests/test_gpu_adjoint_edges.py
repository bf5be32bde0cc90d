"""The adjoint's lattice kernels take 32-node groups, those of the step's
stencil set apart from the others, and its triangles a product differentiated
by hand: odd extents (a last group that is partly past the lattice, rows that
break inside groups), a lattice that is nearly all stencil set, segments of
odd and unequal length, against the oracle's dual numbers."""
import numpy as np
import pytest

import oracle
from paper_1110_0995_gb300 import scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("dims,cells,every", [
    ((37, 21, 19), ["rbc"], 60),              # 14,763 nodes: 11 past a multiple of 32
    ((37, 23, 19), ["rbc"], 7),               # nine segments, eight of odd length, the last one of 4
    ((24, 20, 16), ["rbc"], 25),              # most groups in the stencil set
    ((71, 33, 21), ["rbc", "rbc"], 13),       # a second cell that is not the objective
])
def test_gradient_on_ragged_lattices(dims, cells, every):
    from paper_1110_0995_gb300 import lbibm

    T = 60
    rng = np.random.default_rng(sum(dims))
    bead = np.array([[0.5 * dims[0] + 8.0, 0.5 * dims[1] + 1.0, 0.5 * dims[2] - 1.0, 2.0]], np.float32)
    meshes = scene.place_cells(rng, dims, (1, 0, 0), bead, cells, scene.STABLE, x_range=(0.0, float(bead[0, 0]) - 2.0))
    sc = scene.Scene("adjoint", dims, body_force=(1e-4, 0.0, 0.0), periodic=(1, 0, 0), spheres=bead, meshes=meshes)
    bare = scene.Scene("adjoint", dims, body_force=sc.body_force, periodic=sc.periodic, meshes=meshes)
    sim = lbibm.Simulation.from_scene(bare)
    sim.set_brinkman(bead.astype(np.float64))
    got = sim.adjoint(T, ckpt_every=every, objective_mesh=0)
    ref = oracle.DiffProblem.from_scene(sc)
    want = np.array([ref.run(T, 0, ("bead", k))[1] for k in range(3)])
    # the gradient's bounds of the stated workload: 1e-3 relative, bead
    # components against the largest
    assert got["J"] == pytest.approx(ref.run(T, 0), rel=1e-5)
    assert np.abs(np.asarray(got["beads"]).ravel() - want).max() <= 1e-3 * np.abs(want).max()
    for name in ("ks", "kb"):
        assert got[name] == pytest.approx(ref.run(T, 0, (name,))[1], rel=1e-3)
