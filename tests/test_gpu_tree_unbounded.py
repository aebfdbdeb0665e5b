"""The trees' node pairs where a box is unbounded (coordinates beyond FP32's range on both
sides, in every dimension): such a box meets every patch of the other mesh and nothing
else, with none, one and two levels above the patches whose rows and columns are no
multiples of a node's 4 x 4 children; and the hits are those of the plain precision."""
import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu

P = torch.tensor([1e39, 2e39, 5e38, 3e39], dtype=torch.float64)
Q = torch.tensor([-2e39, -1e39, -3e39, -6e38], dtype=torch.float64)


def _patches(n, m, periodic):
    return -(-(n if periodic else n - 1) // 8) * -(-(m - 1) // 4)


def _spiked(g, periodic):
    """The sheet with two neighbouring vertices, inside the last patch, far beyond FP32."""
    X = g.X.clone()
    X[:, -2, -3] = P
    X[:, -1, -2] = Q
    return tms.Mesh.from_grid(synth.MeshGrid(X, g.s, periodic))


SIZES = [(20, 11, 21, 9), (357, 187, 357, 187), (3000, 400, 2996, 399)]


@pytest.mark.parametrize("size", SIZES, ids=["none", "one", "two"])
@pytest.mark.parametrize("periodic", [True, False])
def test_unbounded_boxes(size, periodic):
    na, ma, nb, mb = size
    p = synth.build_pair(77, na, ma, nb, mb, stretch="exp", n_folds=3, sites=(max(2, nb // 12 & ~1), max(1, mb // 8)),
                         n_hits=0)
    A = _spiked(p.A, periodic)
    B = _spiked(p.B, periodic)
    far = _spiked(synth.MeshGrid(p.B.X + 1e4, p.B.s, periodic), periodic)
    nA, nB = _patches(na, ma, periodic), _patches(nb, mb, periodic)
    plain = dict(precision=0, narrow_filter=0)
    for kw in (dict(), plain):
        tms.search(A, far, hit_capacity=1 << 17, **kw)
        assert tms.last_stats()["patch_pairs"] == nA + nB - 1
    got, want = [gpu_records(tms.search(A, B, hit_capacity=1 << 17, **kw)) for kw in (dict(), plain)]
    assert all(np.array_equal(got[k], want[k]) for k in want) and (na < 100 or len(want["triA"]) > 0)
