"""A search that cannot have a larger list returns an error, each time it is called, and
leaves nothing of its buffers to later searches."""
import numpy as np
import pytest

import paper_2109_14814_gb300 as tms
import synth
from tests.parity import gpu_records

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("start", [1, 32, 33])
@pytest.mark.parametrize("patch", [0, 1])
def test_growth_that_fails(start, patch):
    p = synth.build_pair(31, 600, 200, 500, 180, stretch="exp", n_folds=3, sites=(32, 8), n_hits=0)
    A, B = tms.Mesh.from_grid(p.A), tms.Mesh.from_grid(p.B)
    kw = dict(patch=patch, hit_capacity=1 << 16)
    want = gpu_records(tms.search(A, B, **kw))
    for _ in range(3):
        with pytest.raises(tms.TmsError) as e:
            tms.search(A, B, inject=start | 64, **kw)
        assert e.value.status == tms.TMS_ERR_CUDA
        got = gpu_records(tms.search(A, B, inject=start, **kw))
        assert all(np.array_equal(got[k], want[k]) for k in want)
