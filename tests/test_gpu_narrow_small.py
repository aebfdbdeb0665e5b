"""The FP32 tests on meshes in small units: scaled by a power of two, down to where products
of three and four of a mesh's edges are subnormal FP32 numbers and vanish, two sheets have
the same hits, whose weights are the same bits."""
import numpy as np
import pytest

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("face_level", [0, 1])
@pytest.mark.parametrize("seed", [11, 12])
def test_small_units(seed, face_level):
    p = synth.build_pair(seed, 320, 150, 300, 140, stretch="exp", n_folds=3, sites=(64, 24), n_hits=0)

    def hits(scale):
        A, B = [tms.Mesh.from_grid(synth.MeshGrid(g.X * scale, g.s, True)) for g in (p.A, p.B)]
        return gpu_records(tms.search(A, B, face_level=face_level, hit_capacity=1 << 17))

    one = hits(1.0)
    assert len(one["triA"]) > 700
    for e in range(20, 62):
        got = hits(2.0 ** -e)
        for k in ("triA", "triB", "z"):
            assert np.array_equal(one[k], got[k]), (e, k)
