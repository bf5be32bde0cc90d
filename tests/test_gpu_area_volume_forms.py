"""ibm_area_volume_noalloc on both sides of its rule (cells of up to 8,192
triangles: one launch; a larger one among them: two) against numpy: one
triangle short of and past the line, many cells, an empty one."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("counts", [[1], [255, 256, 257], [2048, 2049, 0, 2047], [8191], [8192, 3], [8193], [8193, 0, 12],
                                    [40000, 700], [20] * 300])
def test_sums_match_numpy(counts):
    import torch

    from paper_1110_0995_gb300 import lbibm

    rng = np.random.default_rng(len(counts) + counts[0])
    n = sum(counts)
    xyz = rng.uniform(-30.0, 200.0, (n + 2, 3))
    tris = rng.integers(0, n + 2, (n, 3)).astype(np.int32)     # any triangles: the sums need no closed mesh
    start = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    # long double, from the edges: exactly 0 where two corners are one node
    a, b, c = (xyz.astype(np.longdouble)[tris[:, k]] for k in range(3))
    normal = np.cross(b - a, c - a)
    s = 0.5 * np.sqrt((normal * normal).sum(1))
    v = (a * normal).sum(1) / 6.0
    want = [np.array([x[i:j].sum() for i, j in zip(start[:-1], start[1:])]) for x in (s, v)]
    size = [np.array([np.abs(x[i:j]).sum() for i, j in zip(start[:-1], start[1:])]) for x in (s, v)]
    dev = [torch.from_numpy(x).cuda() for x in (xyz, tris, start)]
    out = [torch.full((len(counts),), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2)]
    p = ctypes.c_void_p
    st = lbibm.lib().ibm_area_volume_noalloc(p(dev[0].data_ptr()), p(dev[1].data_ptr()), p(dev[2].data_ptr()),
                                             start.ctypes.data_as(p), len(counts), p(out[0].data_ptr()),
                                             p(out[1].data_ptr()), p(torch.cuda.current_stream().cuda_stream))
    assert st == lbibm.LB_OK
    for got, w, z in zip(out, want, size):
        # FP64 on both sides, other orders: 1e-12 of the summed magnitudes
        assert (np.abs(got.cpu().numpy() - w) <= 1e-12 * z + 1e-300).all()
