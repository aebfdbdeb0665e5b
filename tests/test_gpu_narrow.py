"""The FP32 tests, the block's list and the four-lane FP64 solve against the FP64 solve
of every triangle pair (narrow_filter = 0): the same hits bit for bit, for meshes from
a few triangle pairs to many blocks of them, and for meshes that nearly or wholly
coincide, where the FP32 tests reject little or the systems are singular."""
import numpy as np
import pytest
import torch

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu


def _same(A, B, **kw):
    kw.setdefault("hit_capacity", 1 << 17)
    got = gpu_records(tms.search(A, B, **kw))
    solves = tms.last_stats()["fp64_solves"]
    every = gpu_records(tms.search(A, B, narrow_filter=0, **kw))
    assert solves <= tms.last_stats()["fp64_solves"]
    for k in got:
        assert np.array_equal(got[k], every[k]), k
    return got, solves


@pytest.mark.parametrize("face_level", [0, 1])
@pytest.mark.parametrize("shape", [(3, 2), (5, 3), (8, 5), (17, 9), (40, 31), (96, 48)], ids=str)
@pytest.mark.parametrize("shift", [0.0, 1e-13, 1e-8, 1e-3])
def test_filters_change_no_hit(shape, shift, face_level):
    n, m = shape
    p = synth.build_pair(70 + n, max(n, 8), max(m, 3), max(n, 8), max(m, 3), stretch="exp", n_folds=3,
                         sites=(2, 1), n_hits=0)
    X, s = p.A.X[:, :m, :n].contiguous(), p.A.s[:m].contiguous()
    g = torch.Generator().manual_seed(n)
    Y = X + shift * X.abs().max() * (2.0 * torch.rand(X.shape, dtype=X.dtype, generator=g) - 1.0)
    A = tms.Mesh.from_grid(synth.MeshGrid(X, s, True))
    B = tms.Mesh.from_grid(synth.MeshGrid(Y, s, True))
    _, solves = _same(A, B, face_level=face_level)
    assert solves > 0 or shift == 1e-3


@pytest.mark.parametrize("scale", [1e-4, 1e6, 1e30])
def test_scales(scale):
    p = synth.build_pair(11, 200, 90, 180, 70, stretch="exp", n_folds=3, sites=(16, 8), n_hits=0)
    one, _ = _same(tms.Mesh.from_grid(p.A), tms.Mesh.from_grid(p.B))
    A = tms.Mesh.from_grid(synth.MeshGrid(p.A.X * scale, p.A.s, True))
    B = tms.Mesh.from_grid(synth.MeshGrid(p.B.X * scale, p.B.s, True))
    got, _ = _same(A, B)
    if scale == 1e6:
        assert np.array_equal(one["triA"], got["triA"]) and np.array_equal(one["triB"], got["triB"])
