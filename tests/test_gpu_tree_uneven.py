"""Trees over meshes of very unlike size, in either order: a mesh of many nodes against one of
few takes levels that the number of node pairs alone would not; the same candidates and hits
as the grid, and the flag of meshes that are apart."""
import numpy as np
import pytest

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(1023, 130, 8, 5), (1025, 133, 17, 9), (4096, 257, 20, 14), (70000, 9, 9, 6)],
                         ids=lambda s: "x".join(map(str, s)))
def test_uneven_sizes(size):
    na, ma, nb, mb = size
    p = synth.build_pair(300 + nb, na, ma, nb, mb, stretch="exp", n_folds=3, sites=(2, 1), n_hits=0)
    A, B = tms.Mesh.from_grid(p.A), tms.Mesh.from_grid(p.B)
    far = tms.Mesh.from_grid(synth.MeshGrid(p.B.X + 1e3, p.B.s, True))
    for x, y in ((A, B), (B, A)):
        for kw in (dict(), dict(precision=0, narrow_filter=0)):
            tree = gpu_records(tms.search(x, y, **kw))
            st = tms.last_stats()
            assert not st["empty"]
            grid = gpu_records(tms.search(x, y, patch=0, **kw))
            assert st["candidates"] == tms.last_stats()["candidates"] or kw == {}
            assert all(np.array_equal(tree[k], grid[k]) for k in tree)
    for x, y in ((A, far), (far, A)):
        assert len(tms.search(x, y)) == 0 and tms.last_stats()["empty"]
