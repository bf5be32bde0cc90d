"""ibm_area_volume_noalloc twice in a row with a cell of more than 8,192
triangles among the cells: such calls go through the fixed scratch, and the
second one finds there what the first one left behind.  Other positions, a
cell without triangles in another place; against the FP64 oracle and a context
holding the same meshes, with the bounds of the call on small cells."""
import numpy as np
import pytest

import oracle
from paper_1110_0995_gb300 import scene
from test_zz_no_alloc import _context_area_volume, _deformed, _meshes, _noalloc_area_volume

pytestmark = pytest.mark.gpu


def test_two_calls_through_the_scratch():
    import __graft_entry__

    __graft_entry__.build()
    v, t = scene.icosphere(5)
    assert len(t) > 8192
    big = scene.Mesh("big", scene.quantize(10.0 * v + [24.0, 16.0, 16.0], scene.POS_QUANTUM),
                     np.ascontiguousarray(t, np.int32), scene.STABLE["ctc"])
    small = _meshes()
    meshes = [small[0], big, small[1], small[2]]
    rest = np.array([oracle.mesh_area_volume(m.rest, m.tris)[:2] for m in meshes]).T
    for call, (seed, amp) in enumerate([(1, 0.03), (2, 0.01), (3, 0.05)]):
        pos = _deformed(meshes, seed, amp)
        S, V, empty = _noalloc_area_volume(meshes, pos, empty_after=call)
        So, Vo = np.array([oracle.mesh_area_volume(x, m.tris)[:2] for x, m in zip(pos, meshes)]).T
        assert np.abs(S - So).max() <= 1e-10 * So.max() and np.abs(V - Vo).max() <= 1e-10 * Vo.max()
        assert empty == (0.0, 0.0)
        Sc, Vc = _context_area_volume(meshes, pos)
        assert np.abs(S - Sc).max() <= (2e-8 * rest[0] + 1e-5 * np.abs(Sc - rest[0])).max()
        assert np.abs(V - Vc).max() <= (2e-8 * rest[1] + 1e-5 * np.abs(Vc - rest[1])).max()
