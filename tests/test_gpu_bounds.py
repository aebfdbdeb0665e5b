"""The patch level's boxes, rounded vertices and frames (mixed precision) against the plain
precision with every triangle pair solved: the same hits bit for bit, for meshes at the
edges of the bounds pass's tiles, patches and quarters, and for coordinates that are
small integers (exact in FP32, zeros among them) or outside FP32's normal range."""
import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu


def _same(ga, gb, **kw):
    A, B = tms.Mesh.from_grid(ga), tms.Mesh.from_grid(gb)
    kw["hit_capacity"] = 1 << 17
    got = gpu_records(tms.search(A, B, **kw))
    plain = gpu_records(tms.search(A, B, precision=0, narrow_filter=0, **kw))
    for k in got:
        assert np.array_equal(got[k], plain[k]), k
    return len(got["triA"])


@pytest.mark.parametrize("tile_rows", [4, 8])
@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("n,m", [(3, 2), (4, 3), (5, 4), (8, 5), (9, 6), (12, 7), (33, 8), (127, 9), (128, 10),
                                 (129, 11), (257, 13), (261, 17)])
def test_tile_edges(n, m, periodic, tile_rows):
    p = synth.build_pair(400 + n, max(n, 8), max(m, 3), 60, 40, stretch="exp", n_folds=3, sites=(4, 2), n_hits=0)
    ga = synth.MeshGrid(p.A.X[:, :m, :n].contiguous(), p.A.s[:m].contiguous(), periodic)
    _same(ga, p.B, tile_rows=tile_rows)
    _same(p.B, ga, tile_rows=tile_rows)


PLAIN = dict(precision=0, narrow_filter=0)


# (values of 1e-300: FP32 boxes touch where the plain ones are apart by less than a solve
# resolves, so the reference is the grid's FP32 boxes with every pair solved)
@pytest.mark.parametrize("values,ref", [
    ([-2.0, -1.0, -0.0, 0.0, 1.0, 2.0], PLAIN), ([0.0, 1e-300, -1e-300, 5e-324, 1.0, -1.0], dict(patch=0, narrow_filter=0)),
    ([1e-39, -1e-39, 1e-38, -2e-38, 0.0], PLAIN), ([1e39, -1e39, 3e38, -3e38, 0.0], PLAIN),
    ([-16777217.0, 16777217.0, 0.5, -0.5, 1.0 + 2.0 ** -30], PLAIN), ([-1e39, -2e39, -7e38, -1e300], PLAIN)], ids=str)
def test_special_coordinates(values, ref):
    g = torch.Generator().manual_seed(len(values))
    v = torch.tensor(values, dtype=torch.float64)
    grid = lambda n, m: synth.MeshGrid(v[torch.randint(len(values), (4, m, n), generator=g)],
                                       torch.linspace(0, 1, m, dtype=torch.float64), True)
    A, B = tms.Mesh.from_grid(grid(21, 9)), tms.Mesh.from_grid(grid(19, 11))
    got, want = [set(zip(r["triA"], r["triB"])) for r in (gpu_records(tms.search(A, B, tau=1e-9, hit_capacity=1 << 17, **kw))
                                                          for kw in (dict(), ref))]
    if min(values) < -1e38 and max(values) < 0:
        # one box holds every vertex beyond FLT_MAX: no pair is lost to it
        assert tms.last_stats()["candidates"] > 0 and len(got) >= len(want) > 0
    else:
        assert got == want and len(want) > 100
